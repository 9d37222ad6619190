"""The calls a user of this library makes, as measurable cases.

What the library is used for: every decoder layer of a model gets its transforms learned (hundreds of optimisation
steps over all its matrices), its matrices rounded and packed, its coupled pairs rounded by Algorithm 1; at inference
the activations go through the inverse transforms.  The sizes are those of `cafeq_synth.layer_spec` (256 x 512, and
2B-, 9B- and 27B-shaped layers), of the tests (ragged rows, small blocks, per-channel groups) and of the benchmark
(8192 tokens).  Weights follow the same recipe as `cafeq_synth` (Student-t(4) of standard deviation 1/sqrt(d_in), a few
input channels scaled up; the 256 x 512 matrix Gaussian with outliers), drawn on the device.

    listed()  the named cases           draw(rng)  one more case of the same ranges
    prepare(case, seed) -> state        run(state) -> outputs of one pass
    work(case), tolerance(case)
"""
from __future__ import annotations

import math

import torch

import paper_2511_19705_b200 as cq

DEV = "cuda"


# ------------------------------------------------------------------------------------------------ the cases
def listed():
    return [
        # the bulk of a model's quantisation time: optimisation steps over all problems of a layer (q, k, gate single;
        # v-o and up-down coupled), 9B-shaped, 3 bits; a user's call asks for many steps at once
        _layer("layer_9b", 3584, 4096, 2048, 14336, 256, 256, 3, 128, 15.0, 10),
        # the largest layer of the shapes (27B), with the smaller groups; its attention heads take blocks of 128, so
        # the layer is two calls per pass
        _layer("layer_27b_g64", 4608, 4096, 2048, 36864, 256, 128, 3, 64, 15.0, 4),
        # one coupled pair only (2B-shaped MLP), blocks of 128, 4 bits
        _layer("layer_2b_mlp_pair", 2304, 0, 0, 9216, 128, 128, 4, 128, 10.0, 10),
        # a whole optimisation run (50 gradient-descent steps from its start) on a small matrix: launches and latency
        dict(name="single_small", op="single", d_out=256, d_in=512, k=128, axis="in", bits=4, group=128, optimizer="gd", steps=50),
        # one straight-through forward + backward of Eq. 3 for a caller's own optimiser (9B-shaped q)
        dict(name="proxy_ste", op="proxy", mode="ste", d_out=4096, d_in=3584, k=256, axis="in", bits=3, group=128),
        # one straight-through forward + backward of Eq. 5 (9B-shaped v-o pair, grouped-query heads)
        dict(name="pair_ste", op="pair_ste", h=2048, d1=3584, d3=3584, k=256, replicas=2, bits=3, group=128),
        # final rounding of a learned matrix and its packing (9B-shaped gate)
        dict(name="quantize_gate", op="quantize", d_out=14336, d_in=3584, k=256, axis="in", bits=3, group=128),
        # the same on a shape off the large tiles: odd row count, width not a multiple of 256, small blocks and groups
        dict(name="quantize_ragged", op="quantize", d_out=1501, d_in=1440, k=32, axis="in", bits=4, group=32),
        # plain round-to-nearest to packed codes and back to bf16 weights (2B-shaped down projection)
        dict(name="codec_plain", op="codec", d_out=2304, d_in=9216, bits=4, group=64),
        # Algorithm 1 on the 9B-shaped v-o pair
        dict(name="alg1_vo", op="alg1", h=2048, d1=3584, d3=3584, k=256, replicas=2, bits=3, group=128, iters=1),
        # inference: activations through the inverse blocks, a prefill of 8192 tokens and a decode step of 4
        dict(name="apply_prefill", op="apply", tokens=8192, d_in=2304, k=128, transposed=True),
        dict(name="apply_decode", op="apply", tokens=4, d_in=3584, k=256, transposed=True),
    ]


def _layer(name, d, q, kv, ff, k, kv_k, bits, group, outlier, steps):
    return dict(name=name, op="layer", d=d, q=q, kv=kv, ff=ff, k=k, kv_k=kv_k, bits=bits, group=group, outlier=outlier, steps=steps)


def _log(rng, lo, hi, step=1):
    """A multiple of `step` in [lo, hi], spread over the logarithm."""
    v = math.exp(rng.uniform(math.log(lo), math.log(hi)))
    return max(-(-lo // step), min(hi // step, int(round(v / step)))) * step


def _divisor_group(rng, d, choices):
    ok = [g for g in choices if g == 0 or d % g == 0]
    return rng.choice(ok)


def draw(rng):
    op = rng.choices(["layer", "single", "proxy", "pair_ste", "quantize", "codec", "alg1", "apply"], [5, 3, 3, 1, 4, 2, 1, 3])[0]
    bits = rng.choice([3, 3, 4, 4, 2, 8])
    if op == "layer":
        k = rng.choice([128, 256])
        d, r = _log(rng, 1024, 4608, 256), rng.choice([1, 2, 4])
        kv = _log(rng, 512, 2048, 256)
        part = rng.choice(["all", "all", "mlp", "attention"])
        c = _layer("", d, kv * r if part != "mlp" else 0, kv if part != "mlp" else 0, _log(rng, 2 * d, 6 * d, 256) if part != "attention" else 0,
                   k, rng.choice([k, 128]), rng.choice([3, 4]), rng.choice([64, 128]), rng.choice([1.0, 10.0, 15.0]), rng.randint(1, 8))
        c["steps"] = max(1, min(c["steps"], int(4e9 / work(dict(c, steps=1))["bytes"])))
    elif op == "single":
        k = rng.choice([32, 64, 128, 256])
        axis = rng.choice(["in", "in", "out"])
        d_out = _log(rng, 64, 1536, k if axis == "out" else 1)
        d_in = _log(rng, 256, 2048, max(k, 64))
        c = dict(op=op, d_out=d_out, d_in=d_in, k=k, axis=axis, bits=bits, group=_divisor_group(rng, d_in, [0, 32, 64, 128, 128]),
                 optimizer=rng.choice(["gd", "adam"]), steps=rng.randint(5, 50))
    elif op == "proxy":
        k = rng.choice([64, 128, 256])
        d_in = _log(rng, 256, 4608, rng.choice([k, 256]))
        c = dict(op=op, mode=rng.choice(["ste", "ste", "ste_soft", "eval", "surrogate"]), d_out=_log(rng, 100, 4608), d_in=d_in, k=k, axis="in", bits=bits,
                 group=_divisor_group(rng, d_in, [0, 64, 128, 128]))
    elif op in ("pair_ste", "alg1"):
        k, r = rng.choice([64, 128, 256]), rng.choice([1, 1, 2])
        h = _log(rng, 256, 2048 if op == "pair_ste" else 1024, k)
        c = dict(op=op, h=h, d1=_log(rng, int(1.5 * h), 4608, 128), d3=_log(rng, int(1.5 * h), 4608, 64), k=k, replicas=r, bits=rng.choice([3, 4]), group=64 if h * r % 128 else 128)
        if op == "alg1":
            c["iters"] = 1
    elif op == "quantize":
        k = rng.choice([32, 64, 128, 256])
        axis = rng.choice(["in", "in", "out"])
        d_in = _log(rng, 128, 8192, rng.choice([k, max(k, 32) * 3, 256]) if axis == "in" else 32)
        c = dict(op=op, d_out=_log(rng, 64, 8192, k if axis == "out" else 1), d_in=d_in, k=k, axis=axis, bits=bits, group=_divisor_group(rng, d_in, [0, 32, 64, 128, 128]))
    elif op == "codec":
        d_in = _log(rng, 64, 14336, rng.choice([8, 32, 128]))
        c = dict(op=op, d_out=_log(rng, 5, 9216), d_in=d_in, bits=bits, group=_divisor_group(rng, d_in, [0, 32, 64, 128, 256]))
    else:
        k = rng.choice([32, 64, 128, 256])
        c = dict(op=op, tokens=_log(rng, 1, 16384), d_in=_log(rng, 256, 4608, rng.choice([k, 256])), k=k, transposed=rng.random() < 0.75)
        if k == 32:  # (small blocks belong to small models)
            c["tokens"] = min(c["tokens"], 4096)
    c.pop("name", None)
    return c


# ------------------------------------------------------------------------------------------------ inputs
def _gen(seed, tag):
    g = torch.Generator(device=DEV)
    g.manual_seed(int(seed) * 64 + tag)
    return g


def _weight(gen, d_out, d_in, outlier=15.0):
    """Student-t(4) entries of standard deviation 1/sqrt(d_in); 0.1 % of the input channels times `outlier`."""
    W = torch.empty((d_out, d_in), dtype=torch.bfloat16, device=DEV)
    rows = max(1, (1 << 25) // d_in)
    ch = torch.randint(0, d_in, (max(1, round(0.001 * d_in)),), generator=gen, device=DEV)
    for r0 in range(0, d_out, rows):
        n = min(rows, d_out - r0)
        z = torch.randn((n, d_in), generator=gen, device=DEV)
        e = torch.rand((n, d_in), generator=gen, device=DEV).clamp_(min=1e-7).mul_(torch.rand((n, d_in), generator=gen, device=DEV).clamp_(min=1e-7))
        z.mul_(e.log_().mul_(-0.5).rsqrt_()).mul_(1.0 / math.sqrt(2.0 * d_in))  # chi^2_4 / 4 = -ln(u1 u2) / 2
        z[:, ch] *= outlier
        W[r0:r0 + n] = z.to(torch.bfloat16)
    return W


def _weight_gauss(gen, d_out, d_in):
    """N(0, 0.02^2), 0.5 % of the entries times 20."""
    w = torch.randn((d_out, d_in), generator=gen, device=DEV) * 0.02
    w = torch.where(torch.rand((d_out, d_in), generator=gen, device=DEV) < 0.005, w * 20.0, w)
    return w.to(torch.bfloat16)


def _rotations(gen, nb, k, eps=0.0):
    """Haar rotations (QR of a Gaussian with the signs of R's diagonal), eps > 0: off orthogonality as after some steps."""
    q, r = torch.linalg.qr(torch.randn((nb, k, k), generator=gen, device=DEV, dtype=torch.float64))
    q = q * torch.sign(torch.diagonal(r, dim1=-2, dim2=-1)).unsqueeze(-2)
    if eps:
        q = q + torch.randn((nb, k, k), generator=gen, device=DEV, dtype=torch.float64) * (eps / math.sqrt(k))
    return q.to(torch.float32).contiguous()


def _axis(c):
    return cq.AXIS_IN if c["axis"] == "in" else cq.AXIS_OUT


def _blocks(c):
    return (c["d_in"] if c["axis"] == "in" else c["d_out"]) // c["k"]


def _step_size(W, M, c, axis=cq.AXIS_IN):
    """Gradient-descent step: a hundredth of the first gradient's largest entry."""
    g = cq.cafeq_proxy_loss_fwd_bwd(W, M, bits=c["bits"], group=c["group"], taxis=axis)["gradM"]
    return float(1e-2 / max(float(g.abs().max().item()), 1e-30))


def _layer_problems(c):
    """(singles [(d_out, d_in)], pairs [((h, d1), (d3, rh), k, replicas)]) of a layer case."""
    singles, pairs = [], []
    if c["q"]:
        singles += [(c["q"], c["d"]), (c["kv"], c["d"])]
        pairs.append(((c["kv"], c["d"]), (c["d"], c["q"]), c["kv_k"], c["q"] // c["kv"]))
    if c["ff"]:
        if c["q"]:
            singles.append((c["ff"], c["d"]))
        pairs.append(((c["ff"], c["d"]), (c["d"], c["ff"]), c["k"], 1))
    return singles, pairs


def prepare(case, seed):
    c, op = dict(case), case["op"]
    g = _gen(seed, 1)
    s = dict(c=c, op=op)
    if op == "layer":
        singles, pairs = _layer_problems(c)
        by_k = {}
        for n, m in singles:
            W, M = _weight(g, n, m, c["outlier"]), _rotations(g, m // c["k"], c["k"])
            by_k.setdefault(c["k"], ([], []))[0].append(
                dict(W=W, M=M, bits=c["bits"], group=c["group"],
                     cfg=cq.make_cfg(loss_kind=cq.LOSS_SURROGATE, optimizer=cq.OPT_GD, lr=_step_size(W, M, c))))
        for (h, d1), (d3, rh), k, r in pairs:
            by_k.setdefault(k, ([], []))[1].append(
                dict(W1=_weight(g, h, d1, c["outlier"]), W2=_weight(g, d3, rh, c["outlier"]), M=_rotations(g, h // k, k), bits=c["bits"],
                     group1=c["group"], group2=c["group"], replicas=r,
                     cfg=cq.make_cfg(loss_kind=cq.LOSS_LSE, optimizer=cq.OPT_ADAM, lr=1e-4, beta1=0.1, beta2=0.999, eps=1e-8, lambda_orth=0.1,
                                     lse_t=5.0)))
        s["opts"] = {k: cq.LayerOptimizer(*v, max_steps=c["steps"]) for k, v in by_k.items()}
        for o in s["opts"].values():
            o.prepare()
    elif op == "single":
        s["W"] = _weight_gauss(g, c["d_out"], c["d_in"])
        s["M0"] = _rotations(g, _blocks(c), c["k"])
        adam = c["optimizer"] == "adam"
        s["cfg"] = cq.make_cfg(loss_kind=cq.LOSS_SURROGATE, optimizer=cq.OPT_ADAM if adam else cq.OPT_GD,
                               lr=1e-4 if adam else _step_size(s["W"], s["M0"], c, _axis(c)), beta1=0.9 if adam else 0.1, steps=c["steps"])
    elif op == "proxy":
        s["W"], s["M"] = _weight(g, c["d_out"], c["d_in"]), _rotations(g, _blocks(c), c["k"], 0.1)
        s["offsets"] = torch.rand((c["d_out"], c["d_in"]), generator=g, device=DEV) if c["mode"] == "ste_soft" else None
    elif op in ("pair_ste", "alg1"):
        s["W1"], s["W2"] = _weight(g, c["h"], c["d1"]), _weight(g, c["d3"], c["h"] * c["replicas"])
        s["M"] = _rotations(g, c["h"] // c["k"], c["k"], 0.1)
        if op == "pair_ste":
            s["P"] = cq.cafeq_pair_product(s["W1"], s["W2"], k=c["k"], replicas=c["replicas"])
    elif op == "quantize":
        s["W"], s["T"] = _weight(g, c["d_out"], c["d_in"]), _rotations(g, _blocks(c), c["k"], 0.1)
    elif op == "codec":
        s["W"] = _weight(g, c["d_out"], c["d_in"])
    elif op == "apply":
        s["X"] = torch.randn((c["tokens"], c["d_in"]), generator=g, device=DEV).to(torch.bfloat16)
        s["T"] = _rotations(g, c["d_in"] // c["k"], c["k"], 0.1)
    else:
        raise ValueError(op)
    return s


# ------------------------------------------------------------------------------------------------ one pass
def run(s):
    c, op = s["c"], s["op"]
    if op == "layer":
        out = {}
        for k, o in s["opts"].items():
            o.step(c["steps"])
            # (not the Adam moments: at the rotations' start the penalty's gradient is the direction of a rounding error)
            out[str(k)] = dict(M=o.M, history=[h[:, 0] for h in o.hist], status=o.status)
        return out
    if op == "single":
        M = s["M0"].clone()
        history, status, state = cq.cafeq_optimize_single(s["W"], M, s["cfg"], bits=c["bits"], group=c["group"], taxis=_axis(c))
        return dict(M=M, history=history[:, 0], status=status)
    if op == "proxy":
        kw = dict(bits=c["bits"], group=c["group"], taxis=_axis(c))
        if c["mode"] == "eval":
            o = cq.cafeq_proxy_loss_fwd_bwd(s["W"], s["M"], flags=cq.FLAG_EXACT_LOSS | cq.FLAG_NO_GRAD, **kw)
            return dict(losses=o["losses"], status=o["status"])
        if c["mode"] == "surrogate":
            o = cq.cafeq_proxy_loss_fwd_bwd(s["W"], s["M"], **kw)
            return dict(losses=o["losses"][:1], gradM=o["gradM"], status=o["status"])
        soft = c["mode"] == "ste_soft"
        o = cq.cafeq_proxy_loss_fwd_bwd(s["W"], s["M"], loss_kind=cq.LOSS_L2_STE, offsets=s["offsets"], want_grad_offsets=soft, **kw)
        return dict(losses=o["losses"][:3], gradM=o["gradM"], grad_offsets=o["grad_offsets"], status=o["status"])
    if op == "pair_ste":
        o = cq.cafeq_pair_loss_fwd_bwd(s["W1"], s["W2"], s["M"], bits=c["bits"], group1=c["group"], group2=c["group"], replicas=c["replicas"],
                                       P=s["P"], loss_kind=cq.LOSS_PQE_STE)
        return dict(loss=o["losses"][3], gradM=o["gradM"], status=o["status"])
    if op == "alg1":
        o = cq.cafeq_adaptive_round(s["W1"], s["W2"], s["M"], iters=c["iters"], bits=c["bits"], group1=c["group"], group2=c["group"],
                                    replicas=c["replicas"])
        # The second factor's codes, and the product errors, the last of them that of both factors as returned.  The first
        # factor's codes are left out because they cannot be compared: they are a least-squares fit to codes2, and the few
        # entries of codes2 that lie at a tie (1e-4 to 4e-4 of them, against float64) turn 0.5 to 2.5 % of codes1.
        return {n: o[n] for n in ("codes2", "scales2", "pqe", "status")}
    if op == "quantize":
        codes, scales = cq.cafeq_rtn(s["W"], s["T"], bits=c["bits"], group=c["group"], tblock=c["k"], taxis=_axis(c))
        return dict(codes=codes, packed=cq.cafeq_pack(codes, bits=c["bits"]), scales=scales)
    if op == "codec":
        codes, scales = cq.cafeq_rtn(s["W"], None, bits=c["bits"], group=c["group"])
        packed = cq.cafeq_pack(codes, bits=c["bits"])
        return dict(codes=codes, packed=packed, scales=scales, weight=cq.cafeq_dequant(packed, scales, bits=c["bits"], group=c["group"], d_in=c["d_in"]))
    return cq.cafeq_apply_transform(s["X"], s["T"], trole=cq.APPLY_TT if c["transposed"] else cq.APPLY_T)


# ------------------------------------------------------------------------------------------------ what a pass cannot do without
def work(c):
    op = c["op"]
    if op == "layer":  # per step: every weight once through its transform, the parameters and optimiser states read and written
        singles, pairs = _layer_problems(c)
        by = fl = 0.0
        for n, m in singles:
            by += 2.0 * n * m + 8.0 * m * c["k"]
            fl += 2.0 * c["k"] * n * m + 4.0 * m * c["k"] ** 2
        for (h, d1), (d3, rh), k, r in pairs:
            by += 2.0 * (h * d1 + d3 * rh) + 24.0 * h * k
            fl += 2.0 * k * (h * d1 + d3 * rh) + 6.0 * h * k * k
        return dict(bytes=by * c["steps"], flops=fl * c["steps"])
    if op == "single":  # (the matrix may stay on chip between the steps)
        n, m, k = c["d_out"], c["d_in"], c["k"]
        p = _blocks(c) * k * k
        return dict(bytes=2.0 * n * m + 8.0 * p, flops=c["steps"] * (2.0 * k * n * m + 4.0 * p * k))
    if op == "proxy":
        n, m, k = c["d_out"], c["d_in"], c["k"]
        p = _blocks(c) * k * k
        soft = c["mode"] == "ste_soft"
        products = {"eval": 2, "surrogate": 1, "ste": 5, "ste_soft": 5}[c["mode"]]  # U; M^-1 Delta; M^-T E, E Delta^T, gU W^T
        return dict(bytes=2.0 * n * m + (8.0 * n * m if soft else 0.0) + 8.0 * p, flops=products * 2.0 * k * n * m + 4.0 * p * k)
    if op == "pair_ste":
        h, d1, d3, k, r = c["h"], c["d1"], c["d3"], c["k"], c["replicas"]
        n = h * d1 + d3 * h * r  # U and V, U^ V^ and both its gradients, gradients of M
        return dict(bytes=2.0 * n + 4.0 * d1 * d3 + 8.0 * h * k, flops=4.0 * k * n + 3 * 2.0 * d1 * d3 * h)
    if op == "alg1":
        h, d1, d3, k, r, it = c["h"], c["d1"], c["d3"], c["k"], c["replicas"], c["iters"]
        n = h * d1 + d3 * h * r
        half = lambda d, e: 2.0 * d * h * h + 2.0 * h ** 3 + 2.0 * d * e * h + 2.0 * e * h * h  # noqa: E731  Gram, its inverse, P against the factor, solve
        return dict(bytes=3.0 * n + 4.0 * n / c["group"] + 4.0 * h * k,
                    flops=2.0 * k * n + 2.0 * d1 * d3 * h * r + 2.0 * d1 * d3 * h * (2 * it + 1) + it * (half(d1, d3) + half(d3, d1)))
    if op in ("quantize", "codec"):
        n, m = c["d_out"], c["d_in"]
        grp = c["group"] or m
        out = n * m * (1.0 + c["bits"] / 8.0) + 4.0 * n * m / grp
        if op == "codec":
            return dict(bytes=2.0 * n * m + out + 2.0 * n * m, flops=3.0 * n * m)
        return dict(bytes=2.0 * n * m + out + 4.0 * _blocks(c) * c["k"] ** 2, flops=2.0 * c["k"] * n * m)
    n, m = c["tokens"], c["d_in"]
    return dict(bytes=4.0 * n * m + 4.0 * m * c["k"], flops=2.0 * c["k"] * n * m)


def tolerance(c):
    """Measured against another computation of the same outputs (float64 on the device, the shape-agnostic kernels, the
    per-problem calls instead of the layer call), times about four."""
    op = c["op"]
    n = float(c.get("d_out", 0) * c.get("d_in", 0)) or 1.0
    if op == "codec":
        return "exact"
    if op in ("layer", "single"):  # parameters after up to 10 Adam steps at 1e-4: 1.2e-4 / 5e-3; after 50: 1.4e-4 / 4e-3; losses 1e-5
        return {"rel": 6e-4, "max": 0.03}
    if op == "proxy":  # straight-through: 3.2e-5 / 4e-3 when one code in 1.5e7 falls on the other side of a tie, 1e-6 with no tie
        return {"rel": min(0.03, 3e-4 + 3.5 / math.sqrt(n)), "max": 0.1}
    if op == "pair_ste":  # 2.4e-3 / 0.14 (entries of the inverse on the other side of a bf16 rounding, and codes that follow)
        return {"rel": 1e-2, "max": 0.6}
    if op == "quantize":  # codes 4e-6, scales 3e-7 / 1e-6; a single code more or less on a small matrix
        return {"rel": 2e-6, "max": 1e-5, "differ": min(0.01, 5e-5 + 16.0 / n)}
    if op == "alg1":  # codes2 3.7e-4, scales2 1.7e-4 / 6.3e-3, errors 9e-4
        return {"rel": 4e-3, "max": 0.03, "differ": 1.5e-3}
    return {"rel": 6e-4, "max": 0.01}  # bf16 results: 1.4e-4, one rounding step of 2^-7
