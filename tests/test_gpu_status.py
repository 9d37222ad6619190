"""A status word that an earlier call has raised: the kernels of a later call leave, as whole blocks (a block of which some threads
stay runs into its bounded waits, two seconds each), and parameters keep their values."""
import time

import pytest

import cafeq_synth as syn
from parity_utils import f32_dev, to_dev

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture
def cq(monkeypatch):
    """The binding, with every status word that it makes already raised."""
    import paper_2511_19705_b200 as m
    m.lib()

    class T:
        def __getattr__(self, name):
            return getattr(torch, name)

        def zeros(self, *a, **kw):
            if a and a[0] == 1 and kw.get("dtype") is torch.int32:
                return torch.full((1,), 5, **kw)
            return torch.zeros(*a, **kw)

    monkeypatch.setattr(m, "torch", T())
    return m


def _left(out):
    t = time.perf_counter()
    assert int(out["status"].item()) == 5
    assert time.perf_counter() - t < 1.0


@pytest.mark.parametrize("k", [32, 64, 128, 256])
def test_single_and_pair_steps(cq, k):
    W = to_dev(syn.weight_student_t(192, 512, 3))
    M = f32_dev(syn.perturbed_blocks(512 // k, k, 5, 0.02))
    for kind in (cq.LOSS_SURROGATE, cq.LOSS_L2_STE):
        _left(cq.cafeq_proxy_loss_fwd_bwd(W, M, bits=4, group=128, loss_kind=kind, flags=cq.FLAG_EXACT_LOSS))
    W1 = to_dev(syn.weight_student_t(512, 256, 4))
    P = cq.cafeq_pair_product(W1, W, k=k)
    for kind in (cq.LOSS_LSE, cq.LOSS_PQE_STE):
        _left(cq.cafeq_pair_loss_fwd_bwd(W1, W, M, bits=4, group1=128, group2=128, P=P, loss_kind=kind, lambda_orth=0.1))
    before = M.clone()
    for cfg in (cq.make_cfg(steps=2, optimizer=cq.OPT_ADAM), cq.make_cfg(steps=2)):
        assert int(cq.cafeq_optimize_single(W, M, cfg, bits=4, group=128)[1].item()) == 5 and torch.equal(M, before)


def test_layer_and_rounding(cq):
    k = 128
    W1, W2 = to_dev(syn.weight_student_t(256, 512, 6)), to_dev(syn.weight_student_t(384, 256, 7))
    Ms, Mp = f32_dev(syn.perturbed_blocks(4, k, 5, 0.02)), f32_dev(syn.perturbed_blocks(2, k, 8, 0.02))
    b1, b2 = Ms.clone(), Mp.clone()
    lay = cq.LayerOptimizer([dict(W=W1, M=Ms, bits=4, group=128, cfg=cq.make_cfg())],
                            [dict(W1=W1, W2=W2, M=Mp, bits=4, group1=128, group2=128, cfg=cq.make_cfg(loss_kind=cq.LOSS_LSE, optimizer=cq.OPT_ADAM))], 2)
    lay.step(2)
    _left(dict(status=lay.status))
    assert torch.equal(Ms, b1) and torch.equal(Mp, b2)
    _left(cq.cafeq_adaptive_round(W1, W2, Mp, iters=1, bits=4, group1=128, group2=128))
    status = torch.full((1,), 5, dtype=torch.int32, device="cuda")
    for rows in (4, 256):
        cq.cafeq_apply_transform(W1[:rows], Ms, status=status)
    _left(dict(status=status))
