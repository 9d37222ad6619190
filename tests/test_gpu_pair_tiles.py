"""Blocks of 256 run on CTA pairs where records are made (tiles of 256 rows, output axis: columns) and in the sparse backward (tiles of
128 contraction entries), their codes, residuals and products with activations on one CTA a tile.  Sizes at the edges of those tiles, groups narrower and wider than a CTA's half and straddling it, against the
shape-agnostic kernels."""
import pytest
import torch

pytestmark = pytest.mark.gpu


def _case(d_out, d_in, nb, seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    W = torch.randn((d_out, d_in), generator=g, device="cuda")
    W[:, 5] *= 12.0
    M = torch.linalg.qr(torch.randn((nb, 256, 256), generator=g, device="cuda", dtype=torch.float64))[0]
    return (W / d_in ** 0.5).bfloat16(), M.float().contiguous()


# rows: less than one CTA's half, one more than a half, one tile, one more; columns: one and several blocks, a half tile at the end
@pytest.mark.parametrize("axis,d_out,d_in,group", [
    ("in", 1, 256, 128), ("in", 127, 512, 64), ("in", 129, 256, 128), ("in", 256, 768, 256), ("in", 257, 512, 128), ("in", 700, 1024, 512),
    ("out", 256, 128, 128), ("out", 256, 384, 64), ("out", 512, 640, 128), ("out", 256, 1152, 192), ("out", 512, 768, 384),
    ("out", 768, 1280, 256)])
def test_loss_and_gradient(axis, d_out, d_in, group):
    import paper_2511_19705_b200 as cq
    W, M = _case(d_out, d_in, (d_in if axis == "in" else d_out) // 256, d_out + d_in)
    kw = dict(bits=3, group=group, taxis=cq.AXIS_IN if axis == "in" else cq.AXIS_OUT)
    got = cq.cafeq_proxy_loss_fwd_bwd(W, M, flags=cq.FLAG_EXACT_LOSS, **kw)
    want = cq.cafeq_proxy_loss_fwd_bwd(W, M, flags=cq.FLAG_EXACT_LOSS | cq.FLAG_GENERIC, **kw)
    assert int(got["status"].item()) == 0 and int(want["status"].item()) == 0
    # coefficients as two bf16 terms: 2^-17; the inverse on one side by iteration, on the other by elimination in fp32: 1e-5.  The
    # residual of Eq. 3 is kept in bf16: 2^-9 per entry, independent, so a sum of n squares is off by a few times 2^-9 / sqrt(n).
    assert torch.allclose(got["losses"][0], want["losses"][0], rtol=2e-4)
    assert torch.allclose(got["losses"][1], want["losses"][1], rtol=1e-4 + 8 * 2.0 ** -9 / W.numel() ** 0.5)
    g, w = got["gradM"].double(), want["gradM"].double()
    for b in range(g.shape[0]):
        assert ((g[b] - w[b]).norm() / w[b].norm()).item() <= 5e-4, b


# half a tile of contraction entries at the end of the paired backward on the output axis
@pytest.mark.parametrize("d_out,d_in,group", [(256, 64, 64), (512, 192, 64), (256, 576, 192), (512, 704, 64)])
def test_loss_and_gradient_half_tile(d_out, d_in, group):
    test_loss_and_gradient("out", d_out, d_in, group)


# rows apart by more than their width: the padding holds NaN and must not be met
@pytest.mark.parametrize("axis,d_out,d_in,group,pad", [("in", 300, 512, 128, 8), ("in", 257, 768, 64, 256), ("out", 512, 384, 64, 24),
                                                       ("out", 256, 640, 128, 128)])
def test_padded_rows(axis, d_out, d_in, group, pad):
    import paper_2511_19705_b200 as cq
    W, M = _case(d_out, d_in, (d_in if axis == "in" else d_out) // 256, d_out + d_in)
    wide = torch.full((d_out, d_in + pad), float("nan"), device="cuda", dtype=torch.bfloat16)
    wide[:, :d_in] = W
    kw = dict(bits=3, group=group, taxis=cq.AXIS_IN if axis == "in" else cq.AXIS_OUT)
    for loss in (cq.LOSS_SURROGATE, cq.LOSS_L2_STE):
        got = cq.cafeq_proxy_loss_fwd_bwd(wide[:, :d_in], M, loss_kind=loss, **kw)
        want = cq.cafeq_proxy_loss_fwd_bwd(W, M, loss_kind=loss, **kw)
        assert int(got["status"].item()) == 0
        n = 1 if loss == cq.LOSS_SURROGATE else 3
        assert torch.allclose(got["losses"][:n], want["losses"][:n], rtol=1e-5)
        g, w = got["gradM"].double(), want["gradM"].double()
        assert ((g - w).norm() / w.norm()).item() <= 1e-5  # (the same values, summed in another order)
    c, s = cq.cafeq_rtn(wide[:, :d_in], M, bits=3, group=group, tblock=256, taxis=kw["taxis"])
    cw, sw = cq.cafeq_rtn(W, M, bits=3, group=group, tblock=256, taxis=kw["taxis"])
    assert torch.equal(c, cw) and torch.equal(s, sw)


@pytest.mark.parametrize("tokens,d_in,transposed", [(65, 256, True), (128, 512, False), (257, 768, True), (500, 1024, True)])
def test_apply(tokens, d_in, transposed):
    import paper_2511_19705_b200 as cq
    X, T = _case(tokens, d_in, d_in // 256, tokens)
    y = cq.cafeq_apply_transform(X, T, trole=cq.APPLY_TT if transposed else cq.APPLY_T).double()
    P = T.bfloat16().double()
    P = P.transpose(1, 2) if transposed else P
    ref = torch.einsum("tbj,bij->tbi", X.double().reshape(tokens, -1, 256), P).reshape(tokens, d_in)
    assert ((y - ref).abs() <= ref.abs() * 2.0 ** -8 + 1e-5 * ref.abs().max()).all()


@pytest.mark.parametrize("axis,d_out,d_in", [("in", 130, 512), ("in", 300, 256), ("out", 512, 384)])
def test_codes(axis, d_out, d_in):
    import paper_2511_19705_b200 as cq
    W, T = _case(d_out, d_in, (d_in if axis == "in" else d_out) // 256, 3)
    codes, scales = cq.cafeq_rtn(W, T, bits=4, group=128, tblock=256, taxis=cq.AXIS_IN if axis == "in" else cq.AXIS_OUT)
    P = T.bfloat16().double()
    if axis == "in":
        U = torch.einsum("obj,bij->obi", W.double().reshape(d_out, -1, 256), P).reshape(d_out, d_in)
    else:
        U = torch.einsum("bjc,bij->bic", W.double().reshape(-1, 256, d_in), P).reshape(d_out, d_in)
    x = U.reshape(d_out, -1, 128)
    s = x.abs().amax(-1, keepdim=True) / 7
    q = x / s
    assert torch.allclose(scales.double().reshape(s.shape[:2]), s[..., 0], rtol=1e-5)
    c = codes.double().reshape(x.shape)
    # a code may differ from the rounded quotient only where that lies next to a half-integer: sums of 256 terms in fp32
    assert ((c - q).abs() <= 0.5 + 7 * 2.0 ** -18 * 16).all()


# Weights on a coarse grid under permutations: quotients fall on half-integers everywhere, and those are decided by the division of the
# quantiser without a transform.  Groups of both widths, a half tile of columns and of rows.
@pytest.mark.parametrize("axis,k,d_out,d_in", [("in", 64, 130, 640), ("in", 128, 257, 384), ("in", 256, 200, 768), ("out", 128, 384, 640),
                                               ("out", 256, 512, 896)])
@pytest.mark.parametrize("group", [64, 128])
def test_codes_at_ties(axis, k, d_out, d_in, group):
    import paper_2511_19705_b200 as cq
    g = torch.Generator().manual_seed(6)
    W = (torch.randint(-8, 9, (d_out, d_in), generator=g) / 64.0).bfloat16().cuda()
    n = (d_in if axis == "in" else d_out) // k
    p = torch.stack([torch.randperm(k, generator=g) + b * k for b in range(n)]).reshape(-1)
    T = torch.zeros(n, k, k)
    for b in range(n):
        T[b, torch.arange(k), p[b * k:(b + 1) * k] - b * k] = 1
    U = (W[:, p.cuda()] if axis == "in" else W[p.cuda()]).contiguous()
    want, ws = cq.cafeq_rtn(U, None, bits=3, group=group)
    got, gs = cq.cafeq_rtn(W, T.cuda(), bits=3, group=group, tblock=k, taxis=cq.AXIS_IN if axis == "in" else cq.AXIS_OUT)
    assert torch.equal(got, want) and torch.equal(gs, ws)
    if axis == "in":  # the residual takes the same decisions: straight-through gradient against the shape-agnostic kernels
        kw = dict(bits=3, group=group, loss_kind=cq.LOSS_L2_STE)
        a = cq.cafeq_proxy_loss_fwd_bwd(W, T.cuda(), **kw)["gradM"].double()
        b = cq.cafeq_proxy_loss_fwd_bwd(W, T.cuda(), flags=cq.FLAG_GENERIC, **kw)["gradM"].double()
        assert ((a - b).norm() / b.norm()).item() <= 2.0 ** -14


# Straight-through Eq. 3 with the Gram matrix in parts and the scale path in the product's epilogue: rows off the chunks of 64, off the
# parts, and in the last row tile's first and second half; and sizes below the line of each.  The transforms are permutations in which
# half of the rows also take another's entry: sums of two and an inverse of 0, 1 and -1 are exact, so both sides round the same values.
@pytest.mark.parametrize("d_out,d_in,group", [(1100, 2048, 128), (4200, 512, 64), (4165, 512, 128), (833, 2560, 64), (1030, 1024, 128),
                                              (2113, 256, 64), (250, 512, 128)])
def test_straight_through_gradient(d_out, d_in, group):
    import paper_2511_19705_b200 as cq
    W, _ = _case(d_out, d_in, d_in // 256, d_out)
    g = torch.Generator().manual_seed(4)
    M = torch.zeros(d_in // 256, 256, 256)
    for m in M:
        p = torch.randperm(256, generator=g)
        m[torch.arange(256), p] = 1
        m[torch.arange(128), p[128:]] = torch.where(torch.rand(128, generator=g) < 0.5, 1.0, -1.0)
    M = M.cuda()
    got = cq.cafeq_proxy_loss_fwd_bwd(W, M, bits=3, group=group, loss_kind=cq.LOSS_L2_STE)
    want = cq.cafeq_proxy_loss_fwd_bwd(W, M, bits=3, group=group, loss_kind=cq.LOSS_L2_STE, flags=cq.FLAG_GENERIC)
    assert int(got["status"].item()) == 0 and int(want["status"].item()) == 0
    # two bf16 terms an operand: 2^-16 per entry of a product, in a chain of four of them
    assert torch.allclose(got["losses"][:3], want["losses"][:3], rtol=2.0 ** -14)
    g, w = got["gradM"].double(), want["gradM"].double()
    for b in range(g.shape[0]):
        assert ((g[b] - w[b]).norm() / w[b].norm()).item() <= 2.0 ** -14, b
