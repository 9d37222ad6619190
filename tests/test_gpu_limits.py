"""Sizes, alignments, non-finite values and workspaces at the limits of what the calls accept."""
import ctypes

import numpy as np
import pytest

import cafeq_synth as syn
from oracle import cafeq_oracle as orc
from parity_utils import f32_dev, rel_err, to_dev, w64

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def cq():
    import paper_2511_19705_b200 as m
    m.lib()
    return m


def test_second_factor_of_more_rows_than_a_grid_has_slices(cq):
    """65 600 rows (gridDim.y ends at 65 535): the product, its quantised error, its straight-through gradient, Algorithm 1."""
    h, d1, d3, k = 64, 64, 65600, 64
    W1 = to_dev(syn.weight_student_t(h, d1, 3))
    W2 = to_dev(np.tile(syn.weight_student_t(64, h, 4), (d3 // 64, 1)))
    M = f32_dev(syn.perturbed_blocks(1, k, 5, 0.02))
    P = cq.cafeq_pair_product(W1, W2, k=k)
    P64 = W1.double().T @ W2.double().T
    assert float((P - P64).norm() / P64.norm()) <= 1e-6
    kw = dict(bits=4, group1=64, group2=64)
    # the rows repeat 64 rows 1025 times, so the squared error and its gradient are 1025 times theirs
    small = cq.cafeq_pair_loss_fwd_bwd(W1, W2[:64], M, P=cq.cafeq_pair_product(W1, W2[:64], k=k), loss_kind=cq.LOSS_PQE_STE, **kw)
    out = cq.cafeq_pair_loss_fwd_bwd(W1, W2, M, P=P, loss_kind=cq.LOSS_PQE_STE, **kw)
    assert int(out["status"].item()) == 0
    assert abs(float(out["losses"][3]) / (1025 * float(small["losses"][3])) - 1) <= 1e-5
    # one chain of d3 / 16 = 4100 fp32 additions in the tensor core, 2^-23 each: 5e-4 in each of the two factors' parts
    assert rel_err(out["gradM"].cpu().numpy(), 1025 * small["gradM"].cpu().numpy()) <= 2e-3
    r = cq.cafeq_adaptive_round(W1, W2, M, iters=1, **kw)
    assert int(r["status"].item()) == 0
    U = r["codes1"].double() * r["scales1"].double()  # one group per row
    V = r["codes2"].double() * r["scales2"].double()
    Mc = M.bfloat16().double()[0]
    Minv = torch.from_numpy(orc.round_bf16(orc.block_inverse(Mc.cpu().numpy()[None]))).cuda().double()[0]
    target = (Mc.T @ W1.double()).T @ (W2.double() @ Minv.T).T
    assert abs(float((U.T @ V.T - target).norm()) / float(r["pqe"][2]) - 1) <= 1e-3


def test_more_operator_blocks_than_a_grid_has_slices(cq):
    """65 600 blocks of 64: row and operators repeat every 64 blocks, and so must the codes and scales."""
    W = to_dev(syn.weight_student_t(1, 4096, 3))
    T = f32_dev(syn.perturbed_blocks(64, 64, 5, 0.1))
    codes, scales = cq.cafeq_rtn(W.repeat(1, 1025), T.repeat(1025, 1, 1), bits=4, group=128, tblock=64)
    c0, s0 = cq.cafeq_rtn(W, T, bits=4, group=128, tblock=64)
    assert torch.equal(codes.view(1025, -1), c0.repeat(1025, 1)) and torch.equal(scales.view(1025, -1), s0.repeat(1025, 1))


def test_captured_step_of_a_small_layer(cq):
    """Few enough blocks that every kernel of the step is launched programmatically, with the penalty on its side stream: a graph's
    replays are the steps made one by one."""
    def layer():
        mk = lambda *a: to_dev(syn.weight_student_t(*a, 2, 10.0))  # noqa: E731
        k = 128
        singles = [dict(W=mk(384, 512, 1), M=f32_dev(syn.perturbed_blocks(4, k, 5, 0.02)), bits=4, group=128,
                        cfg=cq.make_cfg(optimizer=cq.OPT_ADAM, lr=1e-4))]
        pairs = [dict(W1=mk(256, 1024, 3), W2=mk(640, 512, 4), M=f32_dev(syn.perturbed_blocks(2, k, 6, 0.02)), bits=4, group1=128, group2=128,
                      replicas=2, cfg=cq.make_cfg(loss_kind=cq.LOSS_LSE, optimizer=cq.OPT_ADAM, lr=1e-4, lambda_orth=0.1))]
        lay = cq.LayerOptimizer(singles, pairs, 3)
        lay.prepare()
        return lay

    a, b = layer(), layer()
    for _ in range(4):
        a.step(3)
    s = torch.cuda.Stream()
    s.wait_stream(torch.cuda.current_stream())
    with torch.cuda.stream(s):
        b.step(3)
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g, stream=s):
            b.step(3)
        for _ in range(3):
            g.replay()
    torch.cuda.synchronize()
    assert int(a.status.item()) == 0 == int(b.status.item())
    for x, y, hx, hy, sx, sy in zip(a.M, b.M, a.hist, b.hist, a.state, b.state):
        assert float(sx[0]) == 12.0 == float(sy[0])
        # An entry whose gradient drowns in the order of the atomic additions moves by up to 1e-4 a step either way: at most 2.4e-3
        # of entries of about 0.09 after twelve.  One in a thousand of them would make a difference of 0.027 * 1e-3 ** 0.5 = 8e-4.
        assert rel_err(x.cpu().numpy(), y.cpu().numpy()) <= 1e-3 and rel_err(hx[:, 0].cpu().numpy(), hy[:, 0].cpu().numpy()) <= 1e-4


@pytest.mark.parametrize("d_out,d_in,k,group", [(512, 128, 64, 64), (256, 256, 64, 16), (64, 128, 64, 128), (300, 192, 64, 64), (4096, 256, 64, 64)])
def test_gradient_with_every_maximum_in_one_column(cq, d_out, d_in, k, group):
    """One outlier channel holds the maximum of every row's group: all records of a block go to one row of its gradient."""
    Wb = syn.weight_student_t(d_out, d_in, 3)
    W64 = w64(Wb)
    W64[:, 70] *= 40.0
    W = torch.from_numpy(W64).cuda().bfloat16()
    M = syn.perturbed_blocks(d_in // k, k, 5, 0.02)
    a = cq.cafeq_proxy_loss_fwd_bwd(W, f32_dev(M), bits=4, group=group)
    W64 = W.double().cpu().numpy()
    f = orc.single_forward(W64, M, 4, group, "in")
    assert rel_err(a["gradM"].cpu().numpy(), orc.single_grad_surrogate(W64, f, group, "in")) <= 1e-4


@pytest.mark.parametrize("h,d1,d3,k,r", [(64, 64, 128, 64, 1), (128, 192, 64, 32, 2)])
def test_product_at_any_float_address(cq, h, d1, d3, k, r):
    """The product is any float array: one that starts 4 bytes off a 16-byte boundary holds the same, and serves as the target."""
    W1, W2 = to_dev(syn.weight_student_t(h, d1, 3)), to_dev(syn.weight_student_t(d3, r * h, 4))
    d1_, d2_ = cq._pair_descs(W1, W2, k, 4, 64, 64, r)
    ws = torch.empty(cq.workspace_size(d1_, d2_), dtype=torch.uint8, device="cuda")
    buf = torch.full((d1 * d3 + 2,), 9.0, device="cuda")
    off = buf[1:-1].view(d1, d3)
    assert off.data_ptr() % 8 == 4
    rc = cq.lib().cafeq_pair_product(ctypes.byref(d1_), cq._p(W1), ctypes.byref(d2_), cq._p(W2), cq._p(off), cq._p(ws),
                                     ctypes.c_size_t(ws.numel()), cq._stream())
    P = cq.cafeq_pair_product(W1, W2, k=k, replicas=r)
    assert rc == 0 and torch.equal(off, P) and float(buf[0]) == 9.0 == float(buf[-1])
    M = f32_dev(syn.perturbed_blocks(h // k, k, 5, 0.02))
    a, b = (cq.cafeq_pair_loss_fwd_bwd(W1, W2, M, bits=4, group1=64, group2=64, replicas=r, P=x, loss_kind=cq.LOSS_PQE_STE) for x in (off, P))
    assert rel_err(a["gradM"].cpu().numpy(), b["gradM"].cpu().numpy()) <= 1e-5 and abs(float(a["losses"][3] / b["losses"][3]) - 1) <= 1e-5


def _call_proxy(cq, W, M, grad, k, group=128):
    d = cq.make_desc(W.shape[0], W.shape[1], 4, group, k, cq.AXIS_IN, cq.APPLY_T, 1, W.stride(0))
    losses, status = torch.zeros(4, device="cuda"), torch.zeros(1, dtype=torch.int32, device="cuda")
    ws = torch.empty(cq.workspace_size(d), dtype=torch.uint8, device="cuda")
    rc = cq.lib().cafeq_proxy_loss_fwd_bwd(ctypes.byref(d), cq._p(W), cq._p(M), None, None, 0, cq.LOSS_SURROGATE, ctypes.c_float(0), 0,
                                           cq._p(losses), cq._p(grad), None, cq._p(status), cq._p(ws), ctypes.c_size_t(ws.numel()), cq._stream())
    assert rc == 0 and int(status.item()) == 0
    return losses


@pytest.mark.parametrize("k", [32, 64, 128, 256])
def test_gradient_at_any_float_address(cq, k):
    """The gradient's array is any float array: one that starts 4 bytes off a 16-byte boundary holds the same."""
    W = to_dev(syn.weight_student_t(192, 512, 3))
    M = f32_dev(syn.perturbed_blocks(512 // k, k, 5, 0.05))
    aligned, buf = torch.empty_like(M), torch.full((M.numel() + 2,), 9.0, device="cuda")
    off = buf[1:-1]
    assert off.data_ptr() % 16 == 4
    _call_proxy(cq, W, M, aligned, k)
    _call_proxy(cq, W, M, off, k)
    assert rel_err(off.cpu().numpy(), aligned.flatten().cpu().numpy()) <= 1e-5 and float(buf[0]) == 9.0 == float(buf[-1])
    # the same for a pair
    W1 = to_dev(syn.weight_student_t(512, 256, 4))
    d1, d2 = cq._pair_descs(W1, W, k, 4, 128, 128, 1)
    ws = torch.empty(cq.workspace_size(d1, d2), dtype=torch.uint8, device="cuda")
    for g in (aligned, off):
        losses, status = torch.zeros(4, device="cuda"), torch.zeros(1, dtype=torch.int32, device="cuda")
        rc = cq.lib().cafeq_pair_loss_fwd_bwd(ctypes.byref(d1), cq._p(W1), ctypes.byref(d2), cq._p(W), cq._p(M), None, cq.LOSS_LSE,
                                              ctypes.c_float(5.0), ctypes.c_float(0.1), 0, cq._p(losses), cq._p(g), cq._p(status),
                                              cq._p(ws), ctypes.c_size_t(ws.numel()), cq._stream())
        assert rc == 0 and int(status.item()) == 0
    assert rel_err(off.cpu().numpy(), aligned.flatten().cpu().numpy()) <= 1e-5 and float(buf[0]) == 9.0 == float(buf[-1])


@pytest.mark.parametrize("k", [32, 64, 128, 256])
@pytest.mark.parametrize("pair", [False, True])
def test_optimiser_state_at_any_float_address(cq, k, pair):
    """The per-problem runs take a state that starts 4 bytes off a 16-byte boundary, and resume from it."""
    W = to_dev(syn.weight_student_t(192, 512, 3))
    W1 = to_dev(syn.weight_student_t(512, 256, 4))
    M0 = f32_dev(syn.perturbed_blocks(512 // k, k, 5, 0.02))
    n = cq.OPT_STATE_HEADER + 3 * M0.numel()
    got = []
    for shift in (0, 1):
        buf = torch.zeros(n + 4, device="cuda")
        state, M = buf[shift:shift + n], M0.clone()
        assert state.data_ptr() % 16 == 4 * shift
        for resume in (0, 1):
            cfg = cq.make_cfg(loss_kind=cq.LOSS_LSE if pair else cq.LOSS_SURROGATE, optimizer=cq.OPT_ADAM, lr=1e-4, beta1=0.9, steps=3, resume=resume)
            if pair:
                h, st, _ = cq.cafeq_optimize_pair(W1, W, M, cfg, bits=4, group1=128, group2=128, opt_state=state)
            else:
                h, st, _ = cq.cafeq_optimize_single(W, M, cfg, bits=4, group=128, opt_state=state)
            assert int(st.item()) == 0
        assert float(buf[:shift].abs().sum()) == 0.0 == float(buf[shift + n:].abs().sum()) and float(state[0]) == 6.0
        got.append((M, state[cq.OPT_STATE_HEADER + 2 * M0.numel():].clone(), h[:, 0]))
    for a, b in zip(*got):  # parameters, the stored inverse, losses
        assert rel_err(a.cpu().numpy(), b.cpu().numpy()) <= 1e-5


@pytest.mark.parametrize("rows", [5, 130])
@pytest.mark.parametrize("value", [float("inf"), float("nan")])
@pytest.mark.parametrize("k", [32, 64, 128])
def test_non_finite_activation_stays_in_its_block(cq, k, value, rows):
    X = to_dev(syn.weight_student_t(rows, 512, 3))
    T = f32_dev(syn.perturbed_blocks(512 // k, k, 5, 0.1))
    clean = cq.cafeq_apply_transform(X, T)
    X[3, 70] = value
    out = cq.cafeq_apply_transform(X, T)
    b = 70 // k
    hit = torch.zeros_like(out, dtype=torch.bool)
    hit[3, b * k:(b + 1) * k] = True
    assert not torch.isfinite(out[hit]).any() and torch.equal(out[~hit], clean[~hit])


@pytest.mark.parametrize("k", [32, 64, 128])
@pytest.mark.parametrize("shift", [1, 2])
def test_weights_and_activations_at_any_address(cq, monkeypatch, k, shift):
    """384 columns of a wider array: the workspace that a call's own size query gives is enough wherever they start."""
    monkeypatch.setattr(cq, "workspace", lambda n, device="cuda": torch.empty(int(n), dtype=torch.uint8, device=device))  # (not a larger one)
    wide = torch.zeros((300, 392), dtype=torch.bfloat16, device="cuda")
    off = wide[:, shift:shift + 384]
    off.copy_(to_dev(syn.weight_student_t(300, 384, 3, 2, 10.0)))
    W = off.contiguous()
    T = f32_dev(syn.perturbed_blocks(384 // k, k, 5, 0.1))
    a, b = cq.cafeq_apply_transform(off, T), cq.cafeq_apply_transform(W, T)
    assert rel_err(a.float().cpu().numpy(), b.float().cpu().numpy()) <= 1e-3  # (sums in another order, then bf16)
    for group in (64, 128):
        (c1, s1), (c2, s2) = (cq.cafeq_rtn(x, T, bits=4, group=group, tblock=k) for x in (off, W))
        assert float((c1 != c2).float().mean()) <= 1e-4 and rel_err(s1.cpu().numpy(), s2.cpu().numpy()) <= 1e-6
    M1, M2 = T.clone(), T.clone()
    cfg = cq.make_cfg(steps=2, lr=1e-3)
    (h1, st1, _), (h2, st2, _) = (cq.cafeq_optimize_single(x, m, cfg, bits=4, group=128) for x, m in ((off, M1), (W, M2)))
    assert int(st1.item()) == 0 == int(st2.item()) and rel_err(h1[:, 0].cpu().numpy(), h2[:, 0].cpu().numpy()) <= 1e-5


@pytest.mark.parametrize("bad", [float("nan"), float("inf"), -float("inf")])
@pytest.mark.parametrize("k,group", [(64, 128), (64, 64), (128, 64), (256, 128)])
def test_rounding_beside_a_non_finite_block(cq, k, group, bad):
    """A non-finite weight spoils its block of its row.  A group that also covers another block takes its maximum over the values
    that are numbers; the codes of those are the ones of that maximum, and what is not a number is coded -qmax."""
    W = to_dev(syn.weight_student_t(130, 512, 3))
    T = f32_dev(syn.perturbed_blocks(512 // k, k, 5, 0.1))
    c0, s0 = cq.cafeq_rtn(W, T, bits=4, group=group, tblock=k)
    U = cq.cafeq_apply_transform(W, T).float()
    W[3, 70] = bad
    c1, s1 = cq.cafeq_rtn(W, T, bits=4, group=group, tblock=k)
    b, rows = 70 // k, [r for r in range(130) if r != 3]
    assert torch.equal(c1[rows], c0[rows]) and torch.equal(s1[rows], s0[rows])
    touched = {c // group for c in range(b * k, (b + 1) * k)}
    for G in range(512 // group):
        g = slice(G * group, (G + 1) * group)
        if G not in touched:
            assert torch.equal(c1[3, g], c0[3, g]) and s1[3, G] == s0[3, G]
        elif bad != bad and group > k:  # half of the group is numbers
            keep = torch.tensor([c for c in range(G * group, (G + 1) * group) if c // k != b], device="cuda")
            lost = torch.tensor([c for c in range(G * group, (G + 1) * group) if c // k == b], device="cuda")
            m = float(U[3, keep].abs().max())
            assert abs(float(s1[3, G]) * 7 / m - 1) <= 2.0 ** -7
            assert (c1[3, keep].abs().max() == 7) and (c1[3, lost] == -7).all()
        elif bad != bad:  # nothing left: no maximum, codes 0
            assert float(s1[3, G]) == 0.0 and not c1[3, g].any()
        else:
            assert not torch.isfinite(s1[3, G])


@pytest.mark.parametrize("k,nb", [(128, 3), (256, 2), (256, 150), (48, 2), (100, 2), (50, 2), (512, 1)])
def test_elimination_of_any_block(cq, k, nb):
    """Blocks far from orthogonal: the iteration's fall-back inside its own kernel (128, 256) and the kernel of the other sizes, four
    values at a time or (50) one."""
    rng = np.random.default_rng(k)
    M = rng.standard_normal((min(nb, 3), k, k)).astype(np.float32)
    M = np.tile(orc.round_bf16(M).astype(np.float32), (-(-nb // len(M)), 1, 1))[:nb]
    W = torch.zeros((32, nb * k), dtype=torch.bfloat16, device="cuda")
    out = cq.cafeq_proxy_loss_fwd_bwd(W, f32_dev(M), bits=4, group=0, flags=cq.FLAG_NO_GRAD, want_minv=True)
    assert int(out["status"].item()) == 0
    X = out["Minv"].cpu().numpy().astype(np.float64)
    for b in range(min(nb, 3)):
        ref = np.linalg.inv(M[b].astype(np.float64))
        # backward error of elimination: k 2^-24 times the condition number (growth under partial pivoting is small)
        assert np.linalg.norm(X[b] - ref, 2) <= 4 * k * 2.0 ** -24 * np.linalg.cond(M[b].astype(np.float64)) * np.linalg.norm(ref, 2)
        assert all(np.array_equal(X[c], X[b]) for c in range(b, nb, min(nb, 3)))


@pytest.mark.parametrize("k,d_in", [(32, 14336), (64, 14336), (128, 8192), (256, 3584), (256, 8192), (96, 9600)])
@pytest.mark.parametrize("rows", [8, 9, 24, 32, 64])
def test_apply_few_rows_of_any_width(cq, k, d_in, rows):
    """Both sides of the line between the kernel for few rows and the pass over the operators."""
    g = torch.Generator(device="cuda").manual_seed(k + rows)
    X = torch.randn((rows, d_in), device="cuda", generator=g).bfloat16()
    T = torch.randn((d_in // k, k, k), device="cuda", generator=g) * k ** -0.5
    Y = cq.cafeq_apply_transform(X, T).double()
    Tc, Xb = T.bfloat16().double(), X.double().view(rows, d_in // k, k)
    ref = torch.einsum("bij,obj->obi", Tc, Xb).reshape(rows, d_in)
    mag = torch.einsum("bij,obj->obi", Tc.abs(), Xb.abs()).reshape(rows, d_in)
    # half a bf16 step of the result plus the error of k fp32 additions (2^-24 each, on the sum of magnitudes)
    assert ((Y - ref).abs() <= 2.0 ** -8 * ref.abs() + 2.0 ** -24 * k * mag).all()


@pytest.mark.parametrize("k,r,h", [(32, 2, 128), (32, 4, 64), (96, 2, 192), (64, 2, 128), (128, 3, 128)])
def test_replicas_with_any_block_size(cq, k, r, h):
    """The replicas of a factor's blocks are summed before the product: its error is that of fp32 sums for every block size.  h / 16 <= 12
    additions to an accumulator, 2^-24 of a sum that is half of its final size on average: 3.6e-7; the second terms of the sums, added
    first, cost next to nothing."""
    W1, W2 = to_dev(syn.weight_student_t(h, 192, 3)), to_dev(syn.weight_student_t(128, r * h, 4))
    P = cq.cafeq_pair_product(W1, W2, k=k, replicas=r)
    P64 = orc.pair_product(W1.double().cpu().numpy(), W2.double().cpu().numpy(), k, r)
    assert rel_err(P.cpu().numpy(), P64) <= 3.6e-7
    M = syn.perturbed_blocks(h // k, k, 5, 0.02)
    out = cq.cafeq_pair_loss_fwd_bwd(W1, W2, f32_dev(M), bits=4, group1=64, group2=64, replicas=r, P=P, flags=cq.FLAG_EXACT_LOSS)
    f = orc.pair_forward(W1.double().cpu().numpy(), W2.double().cpu().numpy(), M, 4, 64, 64, r, 5.0, 0.0, True)
    assert abs(float(out["losses"][3]) / f["pqe"] ** 2 - 1) <= 1e-3
