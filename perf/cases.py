"""What the library's speed is measured on: calls a program makes through its public entry
points (``mf_meta_grad``, ``mf_inner_rollout``, ``mf_hvp`` and ``mf_dual_gemm_bf16`` by way of
``native``), on shapes of the workloads in ``synth`` and around them.

A case is a dict of plain values.  ``listed()`` names twelve, ``draw(rng)`` makes one more of
the same kinds and ranges; ``prepare`` / ``run`` / ``work`` / ``tolerance`` / ``exact`` take a
case.  Kinds:

* ``meta``     a whole meta-gradient call: rollout, outer gradient, reverse sweep;
* ``rollout``  the inner loop alone (training steps, no second-order work);
* ``hvp``      one Hessian-vector product with the gradient and the per-example tangent
  losses, forward-over-reverse or reverse-over-reverse: one step of the sweep;
* ``gemm``     one dual linear layer (primal and tangent products of a bf16 layer).
"""
from __future__ import annotations

import math

import torch

from paper_2505_00793_gb300 import native, synth

EX, PLR, SLR = synth.EXAMPLE_WEIGHTS, synth.PARAM_LOGLR, synth.SCALAR_LOGLR

# Product-term masks of mf_dual_gemm_bf16: the terms, each (accumulator, A index, B index),
# and the flags of MN-major operands.
TERMS = {1: (0, 0, 0), 2: (0, 1, 0), 4: (0, 0, 1), 8: (1, 1, 0), 16: (1, 0, 1), 32: (0, 1, 1)}
A_MN, B_MN = 1 << 8, 1 << 9

# A float64 evaluation is given up to this many floating-point operations (a few seconds).
EXACT_FLOPS = 5e12


def _mlp(name, kind, dims, act, loss, precision, B, **kw):
    c = dict(name=name, kind=kind, arch="mlp", act=act, loss=loss, precision=precision, B=B,
             T=1, B_outer=B, alpha=0.05, momentum=0.0, optimizer="sgd", adam_eps=1e-3,
             meta_kind=EX, rr=False, bias=True, chain=0, n_layers=len(dims) - 1)
    c.update({f"d{i}": n for i, n in enumerate(dims)})
    c.update(kw)
    return c


def _dec(name, kind, d, heads, ff, blocks, vocab, seq, precision, B, **kw):
    c = dict(name=name, kind=kind, arch="decoder", d=d, heads=heads, ff=ff, blocks=blocks,
             vocab=vocab, seq=seq, precision=precision, B=B, T=1, B_outer=B, alpha=1e-3,
             momentum=0.0, optimizer="sgd", adam_eps=1e-6, meta_kind=EX, rr=False)
    c.update(kw)
    return c


def listed():
    return [
        # The smallest call in earnest: the tiny float32 regression workload, whole.  Nothing
        # but launches and their latency.
        _mlp("mlp_tiny_meta", "meta", [16, 32, 1], "tanh", "squared", "fp32", 8, T=4, alpha=0.1),
        # A float32 step at a size people train MLPs at, with widths and a batch that divide
        # no tile: the precision a user picks to check a result or a derivative.
        _mlp("mlp_fp32_hvp", "hvp", [784, 1023, 1023, 500, 10], "gelu", "ce", "fp32", 500),
        # The wide workload whole: 256-row bf16 layers, 16 inner steps, many small products.
        _mlp("mlp_wide_meta", "meta", [1024] * 5 + [10], "gelu", "ce", "bf16", 256, T=16,
             B_outer=1024),
        # The deep workload's layers and batch over a short horizon: per-parameter learning
        # rates and momentum, where the parameter-sized passes weigh as much as the products.
        _mlp("mlp_deep_meta", "meta", [4096] * 9, "silu", "squared", "bf16", 512, T=2,
             momentum=0.9, meta_kind=PLR),
        # Reverse-over-reverse on ragged bf16 layers: the standard-AD baseline's step.
        _mlp("mlp_rr_hvp", "hvp", [1000, 1537, 1161, 10], "tanh", "ce", "bf16", 300, rr=True),
        # The motivating example of Section 3 (a linear map and an elementwise recursion);
        # the meta-gradient is that of the initial point.
        _mlp("toy_meta", "meta", [4096, 4096], "ident", "chain_mse", "bf16", 1024, T=2,
             alpha=1e-3, meta_kind=0, bias=False, chain=3),
        # The small transformer with its batch and sequence length, two inner steps.
        _dec("dec_small_meta", "meta", 512, 8, 2048, 6, 8192, 256, "bf16", 16, T=2),
        # The larger transformer (the benchmark's workload) over four of its sixteen inner
        # steps, with its momentum and scalar learning rate: the largest call.
        _dec("dec_large_meta", "meta", 1024, 16, 4096, 12, 32768, 1024, "bf16", 8, T=4,
             momentum=0.9, meta_kind=EX | SLR),
        # Two of the larger transformer's blocks and its head, one step of the sweep on two
        # sequences: what one step costs at a small batch.
        _dec("dec_large_hvp", "hvp", 1024, 16, 4096, 2, 32768, 1024, "bf16", 2),
        # A transformer whose heads are 96 wide and whose sequences fill no tile.
        _dec("dec_odd_hvp", "hvp", 768, 8, 2000, 4, 5000, 200, "bf16", 6),
        # A float32 transformer trained for four Adam steps.
        _dec("dec_fp32_rollout", "rollout", 256, 4, 1024, 4, 2048, 128, "fp32", 8, T=4,
             optimizer="adam", meta_kind=EX),
        # One dual linear layer on ragged sizes: the forward product and its tangent.
        dict(name="gemm_dual", kind="gemm", arch="gemm", M=2000, N=3000, K=1000,
             terms=1 | 8 | 16),
    ]


# ---- drawn cases ---------------------------------------------------------------------------

def _log(rng, lo, hi, step=1):
    """A size in [lo, hi], spread over its logarithm, a multiple of ``step``."""
    v = math.exp(rng.uniform(math.log(lo), math.log(hi)))
    return max(lo, min(hi, int(round(v / step)) * step))


def _draw_mlp(rng, precision):
    kind = rng.choice(["meta", "meta", "hvp", "hvp", "rollout"])
    n = rng.randint(1, 5)
    top = 2048 if precision == "fp32" else 4096
    dims = [_log(rng, 16, top, 8)] + [_log(rng, 16, top) for _ in range(n - 1)]
    loss = rng.choice(["squared", "ce"])
    dims.append(_log(rng, 2, 1000) if loss == "ce" else _log(rng, 1, 512))
    adam = rng.random() < 0.25
    meta_kind = rng.choice([EX, PLR, EX | SLR])
    return _mlp("", kind, dims, rng.choice(["tanh", "gelu", "silu"]), loss, precision,
                _log(rng, 8, 1024), T=_log(rng, 1, 12) if kind != "hvp" else 1,
                B_outer=_log(rng, 8, 1024), momentum=0.0 if adam else rng.choice([0.0, 0.9]),
                optimizer="adam" if adam else "sgd", alpha=1e-3 if adam else 0.05,
                meta_kind=meta_kind, rr=kind != "rollout" and rng.random() < 0.25)


def _draw_toy(rng):
    D = _log(rng, 128, 4096, 8)
    return _mlp("", rng.choice(["meta", "hvp"]), [D, D], "ident", "chain_mse", "bf16",
                _log(rng, 64, 1024), T=rng.randint(1, 3), alpha=1e-3, meta_kind=0, bias=False,
                chain=rng.randint(1, 3), rr=rng.random() < 0.3)


def _draw_dec(rng, precision):
    kind = rng.choice(["meta", "hvp", "hvp", "rollout"])
    fp32 = precision == "fp32"
    dh = rng.choice([32, 64] if fp32 else [32, 64, 64, 64, 64, 96, 128])
    heads = _log(rng, 2, (512 if fp32 else 1280) // dh)
    d = dh * heads
    seq = rng.choice([_log(rng, 32, 256 if fp32 else 1024, 8),
                      128 * rng.randint(1, 2 if fp32 else 8)])
    adam = rng.random() < 0.25
    return _dec("", kind, d, heads, _log(rng, 2 * d, 4 * d, 8), rng.randint(1, 6),
                _log(rng, 256, 4096 if fp32 else 32768, 8), seq, precision, rng.randint(1, 12),
                T=rng.randint(1, 4) if kind != "hvp" else 1, B_outer=rng.randint(1, 12),
                momentum=0.0 if adam else rng.choice([0.0, 0.9]),
                optimizer="adam" if adam else "sgd",
                adam_eps=1e-6 if fp32 else 1e-3,
                meta_kind=rng.choice([EX, EX | SLR]),
                rr=kind != "rollout" and rng.random() < 0.25)


def _draw_gemm(rng):
    terms = rng.choice([1, 1 | 8 | 16, 1 | 8 | 16, 2 | 4, 1 | 32])
    M, N, K = _log(rng, 16, 8192, 8), _log(rng, 16, 8192, 8), _log(rng, 64, 8192, 8)
    mn = rng.choice([0, B_MN, A_MN | B_MN])
    if not mn:   # MN-major rows need strides of whole 16 bytes; K-major ones only K
        M, N = M + rng.randint(0, 7), N + rng.randint(0, 7)
    return dict(name="", kind="gemm", arch="gemm", M=M, N=N, K=K, terms=terms | mn)


def draw(rng):
    caps = {"bf16": 25e12, "fp32": 0.15e12}   # about the largest listed case's time
    while True:
        pick = rng.choice(["mlp32", "mlp16", "mlp16", "toy", "dec16", "dec16", "dec32", "gemm"])
        if pick == "gemm":
            c = _draw_gemm(rng)
        elif pick == "toy":
            c = _draw_toy(rng)
        elif pick.startswith("mlp"):
            c = _draw_mlp(rng, "fp32" if pick == "mlp32" else "bf16")
        else:
            c = _draw_dec(rng, "fp32" if pick == "dec32" else "bf16")
        if work(c)["flops"] <= caps[c.get("precision", "bf16")]:
            c.pop("name")
            return c


# ---- inputs --------------------------------------------------------------------------------

def _dims(c):
    return [c[f"d{i}"] for i in range(c["n_layers"] + 1)]


def _workload(c):
    """The ``synth.Workload`` of a case: shapes, optimiser and meta-parameters."""
    kw = dict(alpha=c["alpha"], momentum=c["momentum"], meta_kind=c["meta_kind"],
              optimizer=c["optimizer"], adam_eps=c["adam_eps"])
    if c["arch"] == "decoder":
        w = synth.decoder("case", c["d"], c["heads"], c["ff"], c["blocks"], c["vocab"],
                          c["seq"], B=c["B"], T=c["T"], B_outer=c["B_outer"], **kw)
        return w.with_(precision=c["precision"])
    return synth.Workload("case", _dims(c), c["act"], c["loss"], c["precision"], B=c["B"],
                          T=c["T"], B_outer=c["B_outer"], has_bias=c["bias"],
                          extra={"chain_steps": c["chain"]}, **kw)


def _normal(g, *shape):
    return torch.randn(*shape, generator=g, device="cuda")


def _rand(g, *shape):
    return torch.rand(*shape, generator=g, device="cuda")


def _mlp_theta(c, w, g):
    """Glorot-uniform weights with small biases; the toy's N(0, 1/D) map."""
    dims, parts = _dims(c), []
    for a, b in zip(dims[:-1], dims[1:]):
        if c["loss"] == "chain_mse":
            parts.append(_normal(g, a * b) / math.sqrt(a))
        else:
            parts.append((_rand(g, a * b) * 2 - 1) * math.sqrt(6.0 / (a + b)))
        if c["bias"]:
            parts.append(0.01 * _normal(g, b))
    return torch.cat(parts)


def _dec_theta(w, g):
    """N(0, 0.02) matrices and RMSNorm gains near 1."""
    return torch.cat([1.0 + 0.02 * _normal(g, n) if name.startswith("g") else
                      0.02 * _normal(g, n) for name, n in w.decoder_layout()])


def _zipf(c, g, *shape):
    """Token ids of a Zipf(1.1) law truncated to the vocabulary."""
    p = torch.arange(1, c["vocab"] + 1, device="cuda", dtype=torch.float64) ** -1.1
    u = _rand(g, *shape).double()
    ids = torch.searchsorted(torch.cumsum(p / p.sum(), 0), u, right=True)
    return ids.clamp_(max=c["vocab"] - 1).int()


def _batch(c, w, g, lead, teacher):
    """Inputs and targets of shape [*lead, ...]."""
    if c["arch"] == "decoder":
        ids = _zipf(c, g, *lead, c["seq"] + 1)
        return ids, ids
    dims = _dims(c)
    x = _normal(g, *lead, dims[0])
    if c["precision"] == "bf16":
        x = x.bfloat16()
    if c["loss"] == "ce":
        y = torch.randint(0, dims[-1], lead, generator=g, device="cuda", dtype=torch.int32)
    elif c["loss"] == "chain_mse":
        y = _normal(g, *lead, dims[-1])
    else:   # a network of the same shape with its own weights, and a little noise
        y = _mlp_out(c, teacher, x.float()) + 0.1 * _normal(g, *lead, dims[-1])
    return x.contiguous(), y.contiguous()


def _tensors(c, seed):
    """The inputs of a call, on the GPU, from the seed alone."""
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    if c["kind"] == "gemm":
        M, N, K = c["M"], c["N"], c["K"]
        a = (K, M) if c["terms"] & A_MN else (M, K)
        b = (K, N) if c["terms"] & B_MN else (N, K)
        mk = lambda s: (0.1 * _normal(g, *s)).bfloat16()
        return dict(A0=mk(a), A1=mk(a), B0=mk(b), B1=mk(b))
    w = _workload(c)
    dec = c["arch"] == "decoder"
    t = dict(theta=_dec_theta(w, g) if dec else _mlp_theta(c, w, g))
    teacher = _mlp_theta(c, w, g) if not dec and c["loss"] == "squared" else None
    if c["kind"] == "hvp":
        t["x"], t["y"] = _batch(c, w, g, (c["B"],), teacher)
        # The sweep's tangent is a direction along which the losses change; along a purely
        # random one the tangent losses are sums that cancel, and show only rounding.
        t["v"] = 0.05 * t["theta"] + 1e-3 * _normal(g, t["theta"].numel())
        t["ex_w"] = torch.sigmoid(_normal(g, c["B"]))
        return t
    t["x"], t["y"] = _batch(c, w, g, (c["T"], c["B"]), teacher)
    eta = []
    if c["meta_kind"] & EX:
        eta.append(_normal(g, c["T"] * c["B"]))
    if c["meta_kind"] & PLR:   # per-parameter rates around the constant one
        rate = 1e-2 if c["optimizer"] == "sgd" else c["alpha"]
        eta.append(math.log(rate) + 0.1 * _normal(g, t["theta"].numel()))
    if c["meta_kind"] & SLR:
        eta.append(torch.full((1,), math.log(c["alpha"]), device="cuda"))
    t["eta"] = torch.cat(eta) if eta else None
    if c["kind"] == "meta":
        t["ox"], t["oy"] = _batch(c, w, g, (c["B_outer"],), teacher)
    return t


def prepare(case, seed):
    t = _tensors(case, seed)
    empty = lambda n: torch.empty(n, device="cuda")
    if case["kind"] == "gemm":
        acc = {TERMS[b][0] for b in TERMS if case["terms"] & b}
        t["C0"], t["C1"] = ((torch.empty(case["M"], case["N"], device="cuda") if j in acc else None)
                            for j in (0, 1))
        return dict(case=case, t=t)
    w = _workload(case)
    mf = native.MixFlow.for_workload(w)
    loop = native.loop_desc_for(w, native.MF_HVP_REV_REV if case["rr"] else native.MF_HVP_MIXED_FOR)
    P = t["theta"].numel()
    if case["kind"] == "hvp":
        out = dict(Hv=empty(P), tangent_losses=empty(case["B"]), grad=empty(P))
    elif case["kind"] == "rollout":
        out = dict(theta_T=empty(P))
    else:
        out = dict(d_eta=empty(t["eta"].numel()) if t["eta"] is not None else None,
                   d_theta0=empty(P), outer_loss=empty(1))
    return dict(case=case, t=t, mf=mf, loop=loop, out=out)


def run(state):
    c, t = state["case"], state["t"]
    if c["kind"] == "gemm":
        native.mf_dual_gemm_bf16(c["M"], c["N"], c["K"], t["A0"], t["A1"], t["B0"], t["B1"],
                                 t["C0"], t["C1"], c["terms"])
        return {k: t[k] for k in ("C0", "C1") if t[k] is not None}
    mf, out = state["mf"], state["out"]
    if c["kind"] == "hvp":
        mf.hvp(c["B"], t["theta"], t["x"], t["y"], t["v"], out["Hv"], ex_w=t["ex_w"],
               tangent_losses=out["tangent_losses"], grad=out["grad"],
               hvp_mode=state["loop"].hvp_mode)
    elif c["kind"] == "rollout":
        mf.inner_rollout(state["loop"], t["theta"], t["eta"], t["x"], t["y"], out["theta_T"])
    else:
        mf.meta_grad(state["loop"], t["theta"], t["eta"], t["x"], t["y"], t["ox"], t["oy"],
                     out["d_eta"], out["d_theta0"], out["outer_loss"])
    return {k: v for k, v in out.items() if v is not None}


# ---- the work a call cannot do without -------------------------------------------------------

def _units(c, rows):
    """Flops of one primal product of every linear layer and of the causal attention's two
    products, split into those of the input layer (no data product) and the rest."""
    if c["arch"] == "mlp":
        dims = _dims(c)
        u = [2.0 * rows * a * b for a, b in zip(dims[:-1], dims[1:])]
        return u[0], sum(u[1:]), 0.0
    N, d = rows * c["seq"], c["d"]
    lin = 2.0 * N * (c["blocks"] * (4 * d * d + 2 * d * c["ff"]) + d * c["vocab"])
    return 0.0, lin, 2.0 * N * c["seq"] * d * c["blocks"]


def work(case):
    c = case
    if c["kind"] == "gemm":
        n = sum(1 for b in TERMS if c["terms"] & b)
        used = [TERMS[b] for b in TERMS if c["terms"] & b]
        A, B = ({u[i] for u in used} for i in (1, 2))
        acc = {u[0] for u in used}
        return {"bytes": 2.0 * c["K"] * (c["M"] * len(A) + c["N"] * len(B)) +
                4.0 * c["M"] * c["N"] * len(acc), "flops": 2.0 * c["M"] * c["N"] * c["K"] * n}
    if c["arch"] == "mlp":
        dims = _dims(c)
        P = sum(a * b + (b if c["bias"] else 0) for a, b in zip(dims[:-1], dims[1:]))
        es = 2 if c["precision"] == "bf16" else 4
        row = dims[0] * es + (4 if c["loss"] == "ce" else 4 * dims[-1])
    else:
        d = c["d"]
        P = 2 * c["vocab"] * d + d + c["blocks"] * (2 * d + 4 * d * d + 2 * d * c["ff"])
        row = 4 * (c["seq"] + 1)
    # products per linear layer: forward 1, weight gradient 1, data 1 for a gradient; forward
    # 3, weight tangent 2, data 3 for a dual pass (the input layer has no data product and no
    # input tangent); the attention: 1 pair forward and 2 backward, each three times when dual
    def cost(rows, grad, dual):
        a, b, att = _units(c, rows)
        return grad * (2 * a + 3 * b + 3 * att) + dual * (3 * a + 8 * b + 9 * att)
    n_eta = (c["T"] * c["B"] if c["meta_kind"] & EX else 0) + \
        (P if c["meta_kind"] & PLR else 0) + (1 if c["meta_kind"] & SLR else 0)
    if c["kind"] == "hvp":
        a, b, _ = _units(c, c["B"])
        return {"bytes": 16.0 * P + c["B"] * (row + 8), "flops": cost(c["B"], 0, 1) + a + b}
    if c["kind"] == "rollout":
        return {"bytes": 8.0 * P + 4.0 * n_eta + c["T"] * c["B"] * row,
                "flops": c["T"] * cost(c["B"], 1, 0)}
    return {"bytes": 8.0 * P + 8.0 * n_eta + (c["T"] * c["B"] + c["B_outer"]) * row,
            "flops": c["T"] * cost(c["B"], 1, 1) + cost(c["B_outer"], 1, 0)}


# ---- the same results in float64 -------------------------------------------------------------

def _act(name, z):
    if name == "gelu":
        return torch.nn.functional.gelu(z)
    return {"ident": lambda z: z, "tanh": torch.tanh,
            "silu": lambda z: z * torch.sigmoid(z)}[name](z)


def _mlp_out(c, theta, x):
    dims, o, h = _dims(c), 0, x
    for i, (a, b) in enumerate(zip(dims[:-1], dims[1:])):
        h = h @ theta[o:o + a * b].reshape(a, b)
        o += a * b
        if c["bias"]:
            h = h + theta[o:o + b]
            o += b
        if i + 2 < len(dims):
            h = _act(c["act"], h)
    return h


def _rms(x, g):
    return g * x * torch.rsqrt((x * x).mean(-1, keepdim=True) + 1e-6)


def _dec_out(c, theta, ids):
    d, H, F, V, S = c["d"], c["heads"], c["ff"], c["vocab"], c["seq"]
    dh, B, o = d // H, ids.shape[0], 0

    def take(*shape):
        nonlocal o
        n = math.prod(shape)
        o += n
        return theta[o - n:o].reshape(shape)

    x = take(V, d)[ids[:, :S].long()]
    j = torch.arange(dh // 2, device=x.device, dtype=x.dtype)
    ang = torch.arange(S, device=x.device, dtype=x.dtype)[:, None] * 10000.0 ** (-2 * j / dh)
    cos, sin = torch.cos(ang).repeat(1, 2), torch.sin(ang).repeat(1, 2)

    def rope(q):
        return q * cos + torch.cat([-q[..., dh // 2:], q[..., :dh // 2]], -1) * sin

    mask = torch.ones(S, S, dtype=torch.bool, device=x.device).triu(1)
    for _ in range(c["blocks"]):
        h = _rms(x, take(d)) @ take(d, 3 * d)
        q, k, v = (z.reshape(B, S, H, dh).transpose(1, 2) for z in h.split(d, -1))
        s = (rope(q) @ rope(k).transpose(-1, -2)) / math.sqrt(dh)
        a = torch.softmax(s.masked_fill(mask, -math.inf), -1) @ v
        x = x + a.transpose(1, 2).reshape(B, S, d) @ take(d, d)
        h = _rms(x, take(d)) @ take(d, F)
        x = x + _act("gelu", h) @ take(F, d)
    return _rms(x, take(d)) @ take(d, V)


def _losses(c, theta, x, y):
    """Per-example (per-sequence) losses."""
    if c["arch"] == "decoder":
        f = _dec_out(c, theta, x)
        tgt = x[:, 1:].long()
        return (torch.logsumexp(f, -1) - f.gather(-1, tgt[..., None])[..., 0]).mean(1)
    f = _mlp_out(c, theta, x)
    if c["loss"] == "ce":
        return torch.logsumexp(f, 1) - f.gather(1, y.long()[:, None])[:, 0]
    if c["loss"] == "squared":
        return 0.5 * ((f - y) ** 2).mean(1)
    for i in range(1, c["chain"] + 1):
        f = i * (2.0 + torch.sin(f)) ** torch.cos(f)
    return ((f - y) ** 2).mean(1)


def _exact_gemm(c, t):
    get = lambda n, mn: t[n].double().t() if mn else t[n].double()
    A = [get("A0", c["terms"] & A_MN), get("A1", c["terms"] & A_MN)]
    B = [get("B0", c["terms"] & B_MN), get("B1", c["terms"] & B_MN)]
    out = {}
    for b, (j, ia, ib) in TERMS.items():
        if c["terms"] & b:
            p = A[ia] @ B[ib].t()
            out[f"C{j}"] = out[f"C{j}"] + p if f"C{j}" in out else p
    return out


def _exact_hvp(c, t):
    th = t["theta"].requires_grad_(True)
    w = t["ex_w"].requires_grad_(True)
    l = _losses(c, th, t["x"], t["y"])
    (g,) = torch.autograd.grad((w * l).sum() / c["B"], th, create_graph=True)
    # d <grad L, v> / d theta = H v;  d / d w_b = (grad l_b . v) / B
    Hv, dw = torch.autograd.grad((g * t["v"]).sum(), (th, w))
    return dict(Hv=Hv, tangent_losses=dw * c["B"], grad=g.detach())


def _inner(c, t, theta, state, eta, i, graph):
    """Inner step i: (theta, optimiser state) -> the next ones."""
    o = c["T"] * c["B"] if c["meta_kind"] & EX else 0
    w = torch.sigmoid(eta[i * c["B"]:(i + 1) * c["B"]]) if o else 1.0
    lr = torch.exp(eta[o:]) if eta is not None and eta.numel() > o else c["alpha"]
    L = (w * _losses(c, theta, t["x"][i], t["y"][i])).sum() / c["B"]
    (g,) = torch.autograd.grad(L, theta, create_graph=graph)
    if c["optimizer"] == "sgd":
        m = c["momentum"] * state[0] + g
        return theta - lr * m, (m,)
    m, v = 0.9 * state[0] + 0.1 * g, 0.999 * state[1] + 0.001 * g * g
    r = v / (1 - 0.999 ** (i + 1))
    # sqrt with derivative 0 at 0, where the gradient and both moments are 0
    r = torch.where(r > 0, torch.sqrt(torch.where(r > 0, r, torch.ones_like(r))), 0.0 * r)
    return theta - lr * (m / (1 - 0.9 ** (i + 1))) / (r + c["adam_eps"]), (m, v)


def _exact_loop(c, t):
    n_state = 2 if c["optimizer"] == "adam" else 1
    theta, state = t["theta"], (torch.zeros_like(t["theta"]),) * n_state
    kept = []
    for i in range(c["T"]):
        kept.append((theta, state))
        th, s = _inner(c, t, theta.requires_grad_(True), state, t["eta"], i, False)
        theta, state = th.detach(), tuple(a.detach() for a in s)
    if c["kind"] == "rollout":
        return dict(theta_T=theta)
    theta.requires_grad_(True)
    V = _losses(c, theta, t["ox"], t["oy"]).mean()
    (tb,) = torch.autograd.grad(V, theta)
    sb = (torch.zeros_like(tb),) * n_state
    d_eta = torch.zeros_like(t["eta"]) if t["eta"] is not None else None
    for i in reversed(range(c["T"])):   # pull the cotangents back through one step at a time
        th, st = kept.pop()
        ins = [th.detach().requires_grad_(True)] + [a.detach().requires_grad_(True) for a in st]
        eta = t["eta"].detach().requires_grad_(True) if d_eta is not None else None
        thn, stn = _inner(c, t, ins[0], tuple(ins[1:]), eta, i, True)
        g = torch.autograd.grad((thn, *stn), ins + ([eta] if eta is not None else []),
                                (tb, *sb), allow_unused=True)
        tb = g[0]
        sb = tuple(a if a is not None else torch.zeros_like(tb) for a in g[1:1 + n_state])
        if eta is not None:
            d_eta += g[-1]
    out = dict(d_theta0=tb, outer_loss=V.detach().reshape(1))
    return dict(d_eta=d_eta, **out) if d_eta is not None else out


def exact(case, seed):
    if work(case)["flops"] > EXACT_FLOPS:
        return None
    t = {k: v.double() if v is not None and v.is_floating_point() else v
         for k, v in _tensors(case, seed).items()}
    if case["kind"] == "gemm":
        return _exact_gemm(case, t)
    return _exact_hvp(case, t) if case["kind"] == "hvp" else _exact_loop(case, t)


def tolerance(case):
    """About four times the largest error against ``exact`` seen on the GPU: 6.5e-6 (a
    product's float32 accumulation), 1.5e-6 (float32), 7e-3 (bf16 operands), 9e-3 (bf16
    operands through the toy's recursion)."""
    if case["kind"] == "gemm":
        return {"rel": 3e-5}
    if case["precision"] == "fp32":
        return {"rel": 1e-5}
    return {"rel": 4e-2 if case.get("chain") else 3e-2}
