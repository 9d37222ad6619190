"""CPU checks of the boundary: the library loads, exports every declared symbol, and rejects bad
arguments on the host before anything is launched (no GPU needed for any of this)."""
import ctypes
import os
import re

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


@pytest.fixture(scope="module")
def cq():
    import paper_2511_19705_b200 as m
    from paper_2511_19705_b200 import build
    build.build()
    m.lib()
    return m


def _declared():
    text = open(os.path.join(ROOT, "include", "cafeq.h")).read()
    text = re.sub(r"/\*.*?\*/", "", text, flags=re.S)
    return sorted(set(re.findall(r"\b(cafeq_[a-z0-9_]+)\s*\(", text)))


def test_every_declared_symbol_is_exported(cq):
    names = _declared()
    assert set(names) == set(cq.EXPORTS)
    L = cq.lib()
    for n in names:
        assert getattr(L, n) is not None
    assert cq.version() >= 100
    assert cq.status_string(0) == "ok" and "singular" in cq.status_string(5)


def test_struct_sizes_match_header_layout(cq):
    # uint32 + 2*int32 + (pad) int64 + 7*int32 -> 56 bytes with natural alignment
    assert ctypes.sizeof(cq.MatrixDesc) == 56
    assert ctypes.sizeof(cq.OptCfg) == 52


def test_workspace_size_and_argument_errors(cq):
    d = cq.make_desc(256, 512, 4, 128, 128)
    n = cq.workspace_size(d)
    assert n > 3 * 256 * 512 * 4
    d2 = cq.make_desc(64, 256, 4, 128, 128, cq.AXIS_IN)
    d1 = cq.make_desc(256, 96, 4, 0, 128, cq.AXIS_OUT)
    assert cq.workspace_size(d1, d2) > cq.workspace_size(d1)
    L = cq.lib()
    nb = ctypes.c_size_t(0)
    bad = cq.make_desc(256, 512, 4, 100, 128)            # group does not divide d_in
    assert L.cafeq_workspace_size(ctypes.byref(bad), None, None, ctypes.byref(nb)) == 1
    bad = cq.make_desc(256, 512, 9, 128, 128)            # bits out of range
    assert L.cafeq_workspace_size(ctypes.byref(bad), None, None, ctypes.byref(nb)) == 1
    bad = cq.make_desc(256, 512, 4, 128, 96)             # block does not tile d_in
    assert L.cafeq_workspace_size(ctypes.byref(bad), None, None, ctypes.byref(nb)) == 1
    bad = cq.make_desc(256, 512, 4, 128, 128)
    bad.struct_size = 12
    assert L.cafeq_workspace_size(ctypes.byref(bad), None, None, ctypes.byref(nb)) == 1
    # null pointers are refused before any launch
    z = ctypes.c_void_p(0)
    assert L.cafeq_rtn(ctypes.byref(d), z, z, z, z, z, ctypes.c_size_t(0), z) == 1
    assert L.cafeq_pack(ctypes.byref(d), z, z, z) == 1
    assert L.cafeq_proxy_loss_fwd_bwd(ctypes.byref(d), z, z, z, z, 0, 0, ctypes.c_float(0), 0, z, z, z, z,
                                      ctypes.c_size_t(0), z) == 1


def test_missing_library_fails_loudly(cq, monkeypatch):
    import paper_2511_19705_b200 as m
    monkeypatch.setattr(m, "_lib", None)
    monkeypatch.setattr(m, "LIB_PATH", os.path.join(ROOT, "does_not_exist.so"))
    with pytest.raises(RuntimeError):
        m.lib()


def test_scratch_of_blocks_of_32_is_that_of_any_block(cq):
    """cafeq_rtn's scratch beside the matrix-sized buffers is its operator, once in fp32 and once in bf16, whatever the block size:
    paired blocks need no room of their own (the built-in buffer of cafeq_rtn_noalloc holds what it always held)."""
    for d_out, d_in, axis in ((1, 512, cq.AXIS_IN), (64, 4096, cq.AXIS_IN), (500, 384, cq.AXIS_IN), (1024, 512, cq.AXIS_OUT)):
        for group in (0, 64, 128):
            n = {k: cq.rtn_workspace_size(cq.make_desc(d_out, d_in, 4, group, k, axis), True) for k in (16, 32)}
            dim = d_in if axis == cq.AXIS_IN else d_out
            assert n[32] - n[16] == 6 * dim * 16, (d_out, d_in, axis, group)


def test_apply_scratch_is_two_forms_of_the_operator(cq):
    for k in (32, 64, 256):
        d = cq.make_desc(300, 512, 4, 128, k)
        n = ctypes.c_size_t(0)
        assert cq.lib().cafeq_apply_workspace_size(ctypes.byref(d), ctypes.byref(n)) == 0
        assert n.value <= 1024 + 6 * 512 * k + (300 * 512 * 4 + 256 if k == 32 else 0)


def test_layer_calls_take_the_widths_that_they_state(cq):
    """d_in a multiple of 256 on the input axis; other widths belong to the per-problem calls."""
    for d_in, rc in ((512, 0), (384, 2)):
        p = cq.LayerProblem()
        p.struct_size, p.pair = ctypes.sizeof(cq.LayerProblem), 0
        p.d1 = p.d2 = cq.make_desc(256, d_in, 4, 128, 128)
        p.W1, p.M, p.loss_history, p.cfg = 4096, 4096, 4096, cq.make_cfg()
        n = ctypes.c_size_t(0)
        assert cq.lib().cafeq_layer_workspace_size(ctypes.byref(p), 1, ctypes.byref(n)) == rc


def test_rounding_without_a_transform_asks_for_its_workspace(cq):
    """Groups of 32 / 64 / 128 / 256 need none; every other width is refused without the one that the size query states."""
    p = ctypes.c_void_p(4096)  # (never read: the check comes first)
    for group in (512, 16, 0):
        d = cq.make_desc(8, 512, 4, group)
        need = cq.rtn_workspace_size(d, False)
        assert need > 0
        for ws, n in ((None, 0), (p, need - 256), (ctypes.c_void_p(4100), need)):
            assert cq.lib().cafeq_rtn(ctypes.byref(d), p, None, p, p, ws, ctypes.c_size_t(n), None) == 3
    for group in (32, 64, 128, 256):
        assert cq.rtn_workspace_size(cq.make_desc(8, 512, 4, group), False) == 0
