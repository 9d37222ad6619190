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
    the update, 2^-8 * 1e-3 = 4e-6 from its one-term product, 5e-7 from the rounding of X to fp32 (||X||_F = sqrt(k)).  A
    warm start stops after the update of a residual below 1e-2: 1e-4 + 4e-5."""
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
    assert float(residual(cold, X).max()) <= 1e-5
    for step in (1e-3, 0.2):  # one round, and several
        warm = cold + (step / np.sqrt(k)) * rng.standard_normal(M0.shape).astype(np.float32)
        o = cq.cafeq_proxy_loss_fwd_bwd(W, f32_dev(warm), flags=cq.FLAG_NO_GRAD | cq.FLAG_WARM_MINV, Minv=X.clone(), **kw)
        assert int(o["status"].item()) == 0
        assert float(residual(warm, o["Minv"]).max()) <= 1.5e-4
