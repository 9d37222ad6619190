"""Dense products on CTA pairs (tiles of 256 rows, up to 256 columns, chosen by size) and the pseudo-inverse built from them, at
sizes where tiles end inside the matrix, against float64."""
import pytest
import torch

pytestmark = pytest.mark.gpu


def _weights(h, d1, d3, r, seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    W1 = torch.randn((h, d1), generator=g, device="cuda") / d1 ** 0.5
    W2 = torch.randn((d3, r * h), generator=g, device="cuda") / (r * h) ** 0.5
    W1[:, :: max(1, d1 // 3)] *= 15.0
    return W1.bfloat16(), W2.bfloat16()


def _fold(X, h, k, r):
    return X.reshape(X.shape[0], h // k, r, k).sum(2).reshape(X.shape[0], h)


# one tile; edges inside a tile in both directions; a single row tile; several waves of 74 pairs; replicas
@pytest.mark.parametrize("h,d1,d3,k,r", [(64, 256, 256, 64, 1), (192, 832, 1088, 64, 1), (256, 2368, 192, 128, 2), (320, 4544, 4160, 64, 1),
                                         (1024, 2048, 2304, 256, 2)])
def test_product_against_float64(h, d1, d3, k, r):
    import paper_2511_19705_b200 as cq
    W1, W2 = _weights(h, d1, d3, r, 3)
    P = cq.cafeq_pair_product(W1, W2, k=k, replicas=r).reshape(d1, d3).double()
    ref = W1.double().t() @ _fold(W2.double(), h, k, r).t()
    # fp32 accumulation of h terms: rounding steps of 2^-24 at the accumulator's size add like a walk, sqrt(h) of them at most
    assert ((P - ref).norm() / ref.norm()).item() <= 2.0 ** -24 * h ** 0.5 * 2


def _quant(T, g, bits):
    qm = 2 ** (bits - 1) - 1
    x = T.float().reshape(T.shape[0], -1, g)
    a = x.abs().amax(-1, keepdim=True)
    s = a / torch.full_like(a, qm)
    q = torch.round(x / torch.where(s > 0, s, torch.ones_like(s))).clamp(-qm, qm)
    return q, s, (q * s).reshape(T.shape).double()


# full rank; one row tile of 64; the inner dimension above the outer ones (tall factor); repeated rows and a zero row (the start
# from the Gram matrix is not usable and the iteration restarts)
@pytest.mark.parametrize("h,d1,d3,k,case", [(512, 832, 768, 128, "full"), (64, 192, 256, 64, "full"), (640, 384, 448, 64, "tall"),
                                            (512, 768, 896, 128, "repeated"), (256, 512, 448, 64, "zero")])
def test_first_half_step_against_float64(h, d1, d3, k, case):
    import paper_2511_19705_b200 as cq
    bits, g = 4, 64
    W1, W2 = _weights(h, d1, d3, 1, 5)
    if case == "repeated":
        W1[:3] = W1[k:k + 3]
    if case == "zero":
        W1[7] = 0
    M = torch.eye(k, device="cuda").repeat(h // k, 1, 1)
    o = cq.cafeq_adaptive_round(W1, W2, M, iters=1, bits=bits, group1=g, group2=g)
    assert int(o["status"].item()) in ((0, 6) if case == "tall" else (0,))  # (tall: the second half-step is rank-deficient)
    U, V = W1.double(), W2.double()
    _, _, Uh = _quant(U, g, bits)
    pinv = torch.linalg.pinv(Uh.t(), rtol=1e-10)
    q, s, _ = _quant((pinv @ (U.t() @ V.t())).t(), g, bits)
    s2 = o["scales2"].double().reshape(s.shape[:2])
    # targets carry the condition of Uhat (tens) times 2^-24 sqrt(terms); a code may turn at a rounding tie of that width
    assert ((s2 - s[..., 0]).norm() / s.norm()).item() <= 3e-5
    assert (o["codes2"].double().reshape(q.shape) != q).double().mean().item() <= 1e-4


# The restart from a start that is not usable: what it keeps of the Gram iteration must not leave the row space of the factor.
@pytest.mark.parametrize("h,d1,d3", [(64, 192, 256), (256, 512, 448), (512, 768, 896)])
@pytest.mark.parametrize("case", ["zero", "repeated"])
def test_singular_factor_to_fp32(h, d1, d3, case):
    import paper_2511_19705_b200 as cq
    g = torch.Generator(device="cuda")
    g.manual_seed(1)
    W1 = (torch.randn((h, d1), generator=g, device="cuda") / d1 ** 0.5).bfloat16()
    W2 = (torch.randn((d3, h), generator=g, device="cuda") / h ** 0.5).bfloat16()
    if case == "zero":
        W1[5] = 0
    else:
        W1[0] = W1[40]
    o = cq.cafeq_adaptive_round(W1, W2, None, iters=1, bits=4, group1=64, group2=64, k=64)
    assert int(o["status"].item()) == 0
    _, _, Uh = _quant(W1.double(), 64, 4)
    T = (torch.linalg.pinv(Uh.t(), rtol=1e-10) @ (W1.double().t() @ W2.double().t())).t()
    s = T.reshape(d3, -1, 64).abs().amax(-1) / 7
    # sums of h terms at fp32; 1.2e-7 to 5.5e-7 measured, with four Gram steps kept 3.1e-6 at the repeated row of 64
    assert ((o["scales2"].double() - s).norm() / s.norm()).item() <= 2.0 ** -24 * h ** 0.5


# One row of an otherwise orthonormal factor is weak, so that what is left of the iteration's residual lies in one direction, and with
# W2's first column dominant that direction alone decides scales2, whose exact values are known (the first factor is on its grid, so
# the target is W2).  Over the strengths of the row the residual before the last step passes through all of its range.
def test_residual_in_one_direction():
    import paper_2511_19705_b200 as cq
    H = torch.ones(1, 1)
    while H.shape[0] < 256:
        H = torch.cat([torch.cat([H, H], 1), torch.cat([H, -H], 1)], 0)
    g = torch.Generator().manual_seed(1)
    V = torch.randn(256, 64, generator=g) * 0.01
    V[:, 0] = 1 + torch.rand(256, generator=g)
    W2 = V.bfloat16().cuda()
    want = W2.double()[:, 0] / 127
    for i in range(60):
        W1 = H[:64].clone()
        W1[0] *= 2.0 ** (-3 - i / 12)
        o = cq.cafeq_adaptive_round(W1.bfloat16().cuda(), W2, None, iters=1, bits=8, group1=64, group2=64, k=64)
        assert int(o["status"].item()) == 0
        # the product W1 W2, its two target products and the last step round at fp32: 5.7e-7 with all updates made
        assert ((o["scales2"].double()[:, 0] - want).abs() / want).max().item() <= 11 * 2.0 ** -24, i


# A power of two on either factor changes exponents only.  Its fourth power is far outside fp32 here.
@pytest.mark.parametrize("e1,e2", [(40, 0), (-40, 0), (0, 40), (0, -40), (55, -55), (-55, 55)])
@pytest.mark.parametrize("case", ["full", "zero"])
def test_alternation_at_other_scales(e1, e2, case):
    import paper_2511_19705_b200 as cq
    h, d1, d3, k, g = 256, 512, 448, 64, 64
    W1, W2 = _weights(h, d1, d3, 1, 7)
    if case == "zero":
        W1[7] = 0
    M = torch.eye(k, device="cuda").repeat(h // k, 1, 1)

    def call(A, B):
        o = cq.cafeq_adaptive_round(A, B, M, iters=1, bits=4, group1=g, group2=g)
        assert int(o["status"].item()) == 0
        return o

    want, got = call(W1, W2), call(W1 * 2.0 ** e1, W2 * 2.0 ** e2)
    # (sums that are added atomically may round another way: bounds as against float64 above)
    s, w = got["scales2"].double() * 2.0 ** -e2, want["scales2"].double()
    assert ((s - w).norm() / w.norm()).item() <= 3e-5
    assert (got["codes2"] != want["codes2"]).double().mean().item() <= 1e-4
    p, q = got["pqe"].double() * 2.0 ** -(e1 + e2), want["pqe"].double()
    assert ((p - q).abs() <= 1e-3 * q).all()


def test_same_codes_under_capture():
    import paper_2511_19705_b200 as cq
    h, d1, d3, k = 256, 512, 448, 64
    W1, W2 = _weights(h, d1, d3, 1, 9)
    M = torch.eye(k, device="cuda").repeat(h // k, 1, 1)

    def call():
        return cq.cafeq_adaptive_round(W1, W2, M, iters=1, bits=4, group1=64, group2=64)

    want = call()
    s = torch.cuda.Stream()
    s.wait_stream(torch.cuda.current_stream())
    with torch.cuda.stream(s):
        call()
    torch.cuda.current_stream().wait_stream(s)
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        got = call()
    graph.replay()
    torch.cuda.synchronize()
    assert torch.equal(got["codes1"], want["codes1"]) and torch.equal(got["codes2"], want["codes2"])
    del graph


# one slice of the contraction; several; several and replicas, a row count off the slices; more blocks than half the chip has
@pytest.mark.parametrize("h,d1,d3,k,r", [(256, 256, 320, 256, 2), (512, 1024, 832, 256, 1), (512, 1088, 1600, 256, 2), (768, 2048, 1024, 128, 1),
                                         (9728, 512, 576, 256, 1)])
def test_straight_through_gradient_repeats_itself(h, d1, d3, k, r):
    import paper_2511_19705_b200 as cq
    W1, W2 = _weights(h, d1, d3, r, 11)
    g = torch.Generator(device="cuda")
    g.manual_seed(2)
    M = torch.linalg.qr(torch.randn((h // k, k, k), generator=g, device="cuda"))[0].contiguous()
    P = cq.cafeq_pair_product(W1, W2, k=k, replicas=r)

    def call(flags=0):
        o = cq.cafeq_pair_loss_fwd_bwd(W1, W2, M, bits=3, group1=64, group2=64, replicas=r, P=P, loss_kind=cq.LOSS_PQE_STE, flags=flags)
        assert int(o["status"].item()) == 0
        return o["gradM"]

    want = call()
    for _ in range(4):
        assert torch.equal(call(), want)
    if h <= 768:
        # the shape-agnostic kernels: entries of the inverse and codes on the other side of a rounding (2.4e-3 measured on the 9B shape)
        ref = call(cq.FLAG_GENERIC).double()
        assert ((want.double() - ref).norm() / ref.norm()).item() <= 1e-2
