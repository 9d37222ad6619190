"""Shapes at the edges of the inference kernels' and the tensor-core pass's ranges: few rows, blocks of 32 in pairs or
alone, a last half tile of 128 columns, every code width of the dequantiser."""
import numpy as np
import pytest

import cafeq_synth as syn
from oracle import cafeq_oracle as orc
from parity_utils import assert_codes_tie_aware, f32_dev, rel_err, tie_free_weight, to_dev, w64

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def cq():
    import paper_2511_19705_b200 as m
    m.lib()
    return m


# rows: 1, the rows of one CTA and one more, the most the small kernel takes and one more (k = 32: paired blocks, single blocks)
@pytest.mark.parametrize("rows", [1, 8, 9, 64, 65])
@pytest.mark.parametrize("d_in,k", [(512, 256), (192, 64), (384, 128), (256, 32), (96, 32)])
@pytest.mark.parametrize("transpose", [False, True])
def test_apply_rows(cq, rows, d_in, k, transpose):
    Xb = syn.weight_student_t(rows, d_in, 71, 1, 5.0)
    T = syn.perturbed_blocks(d_in // k, k, 23, 0.2)
    Y = cq.cafeq_apply_transform(to_dev(Xb), f32_dev(T), trole=cq.APPLY_TT if transpose else cq.APPLY_T)
    Y = Y.float().cpu().numpy().astype(np.float64)
    Y64 = orc.inference_apply(w64(Xb), T, "in", transpose)
    A64 = orc.inference_apply(np.abs(w64(Xb)), np.abs(T), "in", transpose)
    # half a bf16 step of the result plus the error of k fp32 additions (2^-24 each, on the sum of magnitudes)
    assert (np.abs(Y - Y64) <= 2.0 ** -8 * np.abs(Y64) + 2.0 ** -24 * k * A64).all()


@pytest.mark.parametrize("bits", [2, 3, 4, 5, 6, 7, 8])
@pytest.mark.parametrize("d_out,d_in,group,ld", [(3, 1040, 8, 1040), (1, 8, 8, 8), (130, 128, 64, 136)])
def test_dequant_every_width(cq, bits, d_out, d_in, group, ld):
    rng = np.random.default_rng(bits)
    qm = 2 ** (bits - 1) - 1
    q = rng.integers(-qm, qm + 1, size=(d_out, d_in)).astype(np.int32)
    s = np.abs(rng.standard_normal((d_out, d_in // group))).astype(np.float32) + 1e-3
    out = cq.cafeq_dequant(torch.from_numpy(orc.pack_codes(q, bits)).cuda(), torch.from_numpy(s).cuda(), bits=bits, group=group, d_in=d_in)
    ref = torch.from_numpy(np.repeat(s, group, axis=1) * q.astype(np.float32)).to(torch.bfloat16)
    assert torch.equal(out.cpu(), ref)
    if ld != d_in:  # a pitch of its own
        import ctypes
        wide = torch.zeros((d_out, ld), dtype=torch.bfloat16, device="cuda")
        d = cq.make_desc(d_out, d_in, bits, group)
        p, sc = torch.from_numpy(orc.pack_codes(q, bits)).cuda(), torch.from_numpy(s).cuda()
        assert cq.lib().cafeq_dequant(ctypes.byref(d), cq._p(p), cq._p(sc), cq._p(wide), ctypes.c_longlong(ld), cq._stream()) == 0
        assert torch.equal(wide[:, :d_in].cpu(), ref) and not wide[:, d_in:].any()


# a half tile at the end (k = 64, 128), paired blocks of 32 with and without one, single blocks of 32 on both axes
@pytest.mark.parametrize("axis,k,group,shape", [("in", 128, 128, (131, 384)), ("in", 64, 64, (70, 640)), ("in", 32, 64, (129, 384)),
                                                ("in", 32, 128, (64, 256)), ("in", 32, 32, (131, 1440)), ("in", 32, 0, (5, 96)),
                                                ("out", 32, 64, (160, 192)), ("out", 32, 0, (96, 40))])
@pytest.mark.parametrize("transposed", [False, True])
def test_rtn_edges(cq, axis, k, group, shape, transposed):
    Wb = syn.weight_student_t(*shape, 31, 2, 10.0)
    T = syn.perturbed_blocks((shape[1] if axis == "in" else shape[0]) // k, k, 9, 0.2)
    codes, scales = cq.cafeq_rtn(to_dev(Wb), f32_dev(T), bits=4, group=group, tblock=k, taxis=cq.AXIS_IN if axis == "in" else cq.AXIS_OUT,
                                 trole=cq.APPLY_TT if transposed else cq.APPLY_T)
    Tc = orc.round_bf16(T)
    U = orc.apply_blocks(w64(Wb), np.transpose(Tc, (0, 2, 1)) if transposed else Tc, axis)
    # (as many codes within the window of a tie as a uniform quotient gives on so few of them)
    assert_codes_tie_aware(codes.cpu().numpy(), scales.cpu().numpy(), orc.quant_sym(U, 4, group), U, group, max_frac=max(1e-4, 2.0 / U.size))


# straight-through gradients through the residual's split: rows that are no multiple of the contraction chunk, a last half tile
@pytest.mark.parametrize("k,group,shape", [(128, 128, (131, 384)), (64, 64, (65, 128)), (256, 64, (7, 512))])
def test_ste_edges(cq, k, group, shape):
    M = syn.perturbed_blocks(shape[1] // k, k, 19, 0.1)
    Wb = tie_free_weight(lambda i: syn.weight_student_t(*shape, seed=77 + 1000 * i, n_outlier_channels=2, mult=10.0),
                         lambda W: orc.apply_blocks(W, orc.round_bf16(M), "in"), 4, group, "rows")
    out = cq.cafeq_proxy_loss_fwd_bwd(to_dev(Wb), f32_dev(M), bits=4, group=group, loss_kind=cq.LOSS_L2_STE)
    f = orc.single_forward(w64(Wb), M, 4, group, "in")
    assert abs(out["losses"][1].item() - f["L2"]) <= 1e-4 * f["L2"]
    assert rel_err(out["gradM"].cpu().numpy(), orc.single_grad_ste(w64(Wb), f, 4, group, "in")) <= 1e-4  # as at whole tiles


# groups as wide as the row: the widest a warp holds, the first a CTA takes, its variants' edges, and beyond (the separate kernels)
@pytest.mark.parametrize("d_out,d_in", [(3, 1024), (3, 1032), (2, 2048), (2, 4104), (2, 8192), (1, 16384), (1, 16392)])
def test_rtn_whole_rows(cq, d_out, d_in):
    Wb = syn.weight_student_t(d_out, d_in, 7, 2, 10.0)
    Q = orc.quant_sym(w64(Wb), 4, 0)
    for T in (None, f32_dev(syn.identity_blocks(d_in, 1))):  # bf16 source; fp32 source (the identity is exact)
        codes, scales = cq.cafeq_rtn(to_dev(Wb), T, bits=4, group=0, tblock=0 if T is None else 1)
        assert np.array_equal(codes.cpu().numpy().astype(np.int32), Q["q"]) and np.array_equal(scales.cpu().numpy(), Q["s"])


# elimination in registers: pivoting across both halves of the rows, exact permutations, the singular block
@pytest.mark.parametrize("k", [32, 64])
def test_small_inverse(cq, k):
    rng = np.random.default_rng(k)
    nb = 6
    M = rng.standard_normal((nb, k, k))
    M[0] = np.eye(k)[::-1]                                   # every pivot off the diagonal
    M[1] = np.eye(k)[rng.permutation(k)] * np.where(rng.random(k) < 0.5, -1.0, 1.0)
    M[2] = syn.perturbed_blocks(1, k, 3, 0.1)[0]
    M[3, 0, 0] = 0.0
    M = orc.round_bf16(M.astype(np.float32)).astype(np.float64)
    W = torch.zeros((64, nb * k), dtype=torch.bfloat16, device="cuda")
    for flags in (cq.FLAG_NO_GRAD, cq.FLAG_NO_GRAD | cq.FLAG_GENERIC):
        out = cq.cafeq_proxy_loss_fwd_bwd(W, f32_dev(M), bits=4, group=0, flags=flags, want_minv=True)
        assert int(out["status"].item()) == 0
        X = out["Minv"].cpu().numpy().astype(np.float64)
        for b in range(nb):
            ref = np.linalg.inv(M[b])
            # backward error of elimination: k 2^-24 times the condition number (growth under partial pivoting is small)
            assert np.linalg.norm(X[b] - ref, 2) <= 4 * k * 2.0 ** -24 * np.linalg.cond(M[b]) * np.linalg.norm(ref, 2)
        assert np.array_equal(X[:2], np.linalg.inv(M[:2]))
    M[4, :, 5] = 0.0
    out = cq.cafeq_proxy_loss_fwd_bwd(W, f32_dev(M), bits=4, group=0, flags=cq.FLAG_NO_GRAD)
    assert int(out["status"].item()) == 5                   # singular block


# group widths of every variant of the fused gradient split (one lane's vector to a warp's eight), with and without replicas
@pytest.mark.parametrize("k,r,h,d1,d3,g1,g2", [(64, 1, 128, 256, 192, 32, 32), (64, 2, 256, 256, 128, 256, 512), (64, 4, 256, 1024, 64, 1024, 1024),
                                               (64, 1, 128, 192, 128, 96, 128)])
def test_pair_ste_group_widths(cq, k, r, h, d1, d3, g1, g2):
    import test_gpu_pqe_ste as pqe
    pqe.test_pqe_ste_gradient_matches_oracle(cq, k, r, h, d1, d3, g1, g2, 4, False)
