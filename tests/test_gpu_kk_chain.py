"""Fused chains of k x k products (one CTA per operator block): sizes at the edges of their range."""
import numpy as np
import pytest

import cafeq_synth as syn
from parity_utils import f32_dev

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def cq():
    import paper_2511_19705_b200 as m
    m.lib()
    return m


@pytest.mark.parametrize("k,nb", [(128, 2), (128, 150), (256, 1), (256, 150)])
def test_fused_newton_schulz_residual(cq, k, nb):
    """||I - bf16(M) X||_F per block, in float64.  A cold start stops after the update of a residual below 1e-3: 1e-6 from
    the update, 2^-8 * 1e-3 = 4e-6 from its one-term product; then 5e-7 from the rounding of X to fp32 (||X||_F = sqrt(k))
    and k 2^-24 because R = I - A X cancels against fp32 accumulators of size up to 1 (one rounding, 2^-24, in each of the
    k^2 entries).  A warm start stops after the update of a residual below 1e-2: 1e-4 + 4e-5 instead of the first two."""
    acc = k * 2.0**-24 + 5e-7
    W = torch.zeros((64, nb * k), dtype=torch.bfloat16, device="cuda")
    M0 = syn.haar_blocks(min(nb, 4), k, 11)
    M0 = np.tile(M0, (-(-nb // len(M0)), 1, 1))[:nb]
    rng = np.random.default_rng(k + nb)
    kw = dict(bits=4, group=64)

    def residual(M, X):
        A = f32_dev(M).bfloat16().double()
        return (torch.eye(k, device="cuda", dtype=torch.float64) - A @ X.double()).flatten(1).norm(dim=1)

    cold = M0 + (0.1 / np.sqrt(k)) * rng.standard_normal(M0.shape).astype(np.float32)
    o = cq.cafeq_proxy_loss_fwd_bwd(W, f32_dev(cold), flags=cq.FLAG_NO_GRAD, want_minv=True, **kw)
    X = o["Minv"]
    assert int(o["status"].item()) == 0
    assert float(residual(cold, X).max()) <= 5e-6 + acc
    for step in (1e-3, 0.2):  # one round, and several
        warm = cold + (step / np.sqrt(k)) * rng.standard_normal(M0.shape).astype(np.float32)
        o = cq.cafeq_proxy_loss_fwd_bwd(W, f32_dev(warm), flags=cq.FLAG_NO_GRAD | cq.FLAG_WARM_MINV, Minv=X.clone(), **kw)
        assert int(o["status"].item()) == 0
        assert float(residual(warm, o["Minv"]).max()) <= 1.4e-4 + acc


@pytest.mark.parametrize("k,nb", [(128, 1), (128, 150), (256, 1), (256, 149)])
def test_fused_gradient_through_the_inverse(cq, k, nb):
    """Eq. 4's gradient with the M^-1 path in the fused chain against the shape-agnostic kernels (elimination, fp32
    products).  Three-term products leave 2^-16 per operand; the inverses differ by the cold start's 2e-5."""
    d_in = nb * k if k == 256 else max(nb, 2) * k
    W = torch.randn((70, d_in), device="cuda").bfloat16()
    M = f32_dev(np.tile(syn.perturbed_blocks(2, k, 5, 0.1), (d_in // k // 2 + 1, 1, 1))[:d_in // k])
    kw = dict(bits=4, group=128)
    a = cq.cafeq_proxy_loss_fwd_bwd(W, M, **kw)
    b = cq.cafeq_proxy_loss_fwd_bwd(W, M, flags=cq.FLAG_GENERIC, **kw)
    assert int(a["status"].item()) == 0
    ga, gb = a["gradM"].double().flatten(1), b["gradM"].double().flatten(1)
    assert float(((ga - gb).norm(dim=1) / gb.norm(dim=1)).max()) <= 2e-4


@pytest.mark.parametrize("k,nb", [(128, 1), (128, 150), (256, 1), (256, 149)])
def test_fused_penalty(cq, k, nb):
    """||M M^T - I||_F / sqrt(h) and its gradient (the difference of two calls: the LogSumExp's part cancels up to the
    order of its atomic additions) against float64.  Three-term products: 2^-16 per operand, fp32 sums of k terms."""
    h = nb * k
    W1 = torch.randn((h, 128), device="cuda").bfloat16()
    W2 = torch.randn((64, max(h, 256)), device="cuda").bfloat16()[:, :h].contiguous()
    M = f32_dev(np.tile(syn.perturbed_blocks(2, k, 5, 0.1), (nb // 2 + 1, 1, 1))[:nb])
    lam = 1e4
    kw = dict(bits=4, group1=128, group2=128)
    a = cq.cafeq_pair_loss_fwd_bwd(W1, W2, M, lambda_orth=lam, **kw)
    b = cq.cafeq_pair_loss_fwd_bwd(W1, W2, M, lambda_orth=0.0, **kw)
    assert int(a["status"].item()) == 0
    Md = M.double()
    R = Md @ Md.transpose(1, 2) - torch.eye(k, device="cuda", dtype=torch.float64)
    n = R.norm()
    pen = float(n) / h**0.5
    assert abs(float(a["losses"][2]) - pen) <= 1e-4 * pen and abs(float(b["losses"][2]) - pen) <= 1e-4 * pen
    ref = 2 * lam * (R @ Md) / (n * h**0.5)
    g = (a["gradM"] - b["gradM"]).double()
    assert float((g - ref).norm() / ref.norm()) <= 1e-4
