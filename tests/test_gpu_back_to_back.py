"""Calls without a pause between them, each reading what the one before wrote, in buffers that the allocator hands out again:
the results are those of calls that wait for one another."""
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def cq():
    import paper_2511_19705_b200 as m
    m.lib()
    return m


def _chain(cq, W, T, k, group, wait):
    out = []
    X = W
    for i in range(6):
        X = cq.cafeq_apply_transform(X, T, trole=cq.APPLY_TT if i % 2 else cq.APPLY_T)  # reads the previous weight
        wait()
        codes, scales = cq.cafeq_rtn(X, T if i % 3 else None, bits=4, group=group, tblock=k if i % 3 else 0)
        wait()
        packed = cq.cafeq_pack(codes, bits=4)
        del codes
        wait()
        X = cq.cafeq_dequant(packed, scales, bits=4, group=group, d_in=W.shape[1])
        del packed, scales
        wait()
        out.append(X.clone())
        wait()
    return torch.stack(out)


@pytest.mark.parametrize("rows,d_in,k,group", [(4, 512, 128, 128), (64, 1024, 256, 64), (300, 1024, 64, 64), (2048, 2048, 256, 128),
                                               (300, 1440, 32, 32), (70, 512, 32, 128), (33, 512, 128, 512)])
def test_chained_calls(cq, rows, d_in, k, group):
    g = torch.Generator(device="cuda").manual_seed(rows + k)
    T = torch.linalg.qr(torch.randn((d_in // k, k, k), device="cuda", generator=g))[0].contiguous()
    Ws = [torch.randn((rows, d_in), device="cuda", generator=g).bfloat16() for _ in range(4)]
    ref = [_chain(cq, W, T, k, group, torch.cuda.synchronize) for W in Ws]
    buf = torch.empty_like(Ws[0])
    for rnd in range(8):
        got = []
        for W in Ws:  # one input buffer, new contents
            buf.copy_(W)
            got.append(_chain(cq, buf, T, k, group, lambda: None))
        assert all(torch.equal(a, b) for a, b in zip(got, ref)), rnd


@pytest.mark.parametrize("k", [64, 128])
def test_straight_through_on_changing_weights(cq, k):
    g = torch.Generator(device="cuda").manual_seed(k)
    M = (torch.eye(k, device="cuda") + 0.02 * torch.randn((1024 // k, k, k), device="cuda", generator=g)).contiguous()
    Ws = [torch.randn((256, 1024), device="cuda", generator=g).bfloat16() for _ in range(3)]
    kw = dict(bits=4, group=128, loss_kind=cq.LOSS_L2_STE)
    ref = []
    for W in Ws:
        ref.append(cq.cafeq_proxy_loss_fwd_bwd(W, M, **kw))
        torch.cuda.synchronize()
    buf = torch.empty_like(Ws[0])
    for _ in range(10):
        for W, r in zip(Ws, ref):
            buf.copy_(W)
            o = cq.cafeq_proxy_loss_fwd_bwd(buf, M, **kw)
            # sums through atomic additions: their order is all that may differ
            assert float((o["gradM"] - r["gradM"]).norm() / r["gradM"].norm()) <= 1e-5
            assert float((o["losses"] - r["losses"]).abs().max() / r["losses"].abs().max()) <= 1e-5
