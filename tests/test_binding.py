"""CPU checks of the Python binding: what it hands to the C calls, and how long that lives."""
import ctypes
import gc
import weakref

import pytest

torch = pytest.importorskip("torch")


@pytest.fixture
def cq(monkeypatch):
    import paper_2511_19705_b200 as m
    from paper_2511_19705_b200 import build
    build.build()
    m.lib()
    monkeypatch.setattr(m, "_raw_stream", lambda: 0)
    m._plan.cache_clear()
    yield m
    m._plan.cache_clear()


class _Calls:
    """Stands in for the typed C calls: drops every cached plan, as other threads' shapes may at any time, and then looks whether
    the descriptor that it was given still exists."""

    def __init__(self, cq):
        self.cq, self.args = cq, []

    def __getattr__(self, name):
        def call(desc, *args):
            alive = [weakref.ref(o) for o in gc.get_objects() if isinstance(o, self.cq.MatrixDesc) and ctypes.addressof(o) == desc]
            assert len(alive) == 1
            self.cq._plan.cache_clear()
            gc.collect()
            assert alive[0]() is not None, f"{name}: the descriptor was freed while the call was using it"
            self.args.append((name, args))
            return 0
        return call


class _Codes:  # an int8 CUDA tensor as far as the binding looks
    dtype, is_cuda, shape, device = torch.int8, True, (4, 64), torch.device("cpu")

    def is_contiguous(self):
        return True

    def data_ptr(self):
        return 4096


def test_descriptor_outlives_the_call(cq, monkeypatch):
    calls = _Calls(cq)
    monkeypatch.setattr(cq, "_hot", lambda: calls)
    cq.cafeq_pack(_Codes(), bits=4)
    cq.cafeq_dequant(torch.zeros((4, 32), dtype=torch.uint8), torch.zeros((4, 1)), bits=4, group=64, d_in=64)
    assert [n for n, _ in calls.args] == ["pack", "dequant"]


def test_addresses_in_place_of_tensors(cq, monkeypatch):
    """Arrays whose shape the binding does not need may be given as device addresses, or left out."""
    calls = _Calls(cq)
    monkeypatch.setattr(cq, "_hot", lambda: calls)
    packed = torch.zeros((4, 32), dtype=torch.uint8)
    cq.cafeq_dequant(packed, 8192, bits=4, group=64, d_in=64)
    assert calls.args[-1][1][:2] == (packed.data_ptr(), 8192)
    cq.cafeq_dequant(packed, None, bits=4, group=64, d_in=64)  # (refused by the C call)
    assert calls.args[-1][1][1] in (None, 0)

    class X(_Codes):
        dtype = torch.bfloat16

        def stride(self, i):
            return (64, 1)[i]

    T = torch.zeros((1, 64, 64))
    for status, given in ((None, (None, 0)), (12288, (12288,)), (torch.zeros(1, dtype=torch.int32), None)):
        cq.cafeq_apply_transform(X(), T, status=status)
        assert calls.args[-1][1][3] in (given or (status.data_ptr(),))
