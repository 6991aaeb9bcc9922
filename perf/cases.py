"""Performance cases of the FAVOR# library: what its users have it do, through the public binding.

A case is a plain dict.  `kind` says which calls one pass makes:

  step      statistics -> closed-form fit -> attention of one batch (parameters refitted on every batch)
  train     the same, followed by the backward pass for a cotangent dY
  features  the feature map alone, queries and keys (random-feature models, caches of key features)
  pairs     kernel estimates of (x, y) pairs over R feature draws with closed-form and pooled variances
  apply     the unnormalised Gaussian-kernel operator on a point set (kernel classification / regression)
  slice     one rank's share of a sequence spread over ranks: key states, then attention from handed-on states
  host      the whole path on host buffers

Sizes are those of the package's workloads (workloads.py) and of the paper's BERT setup (12 heads, 512 tokens,
M = 256), and generic ragged ones around them.  `layout` "blhd" is what a projection layer hands over: [B, L, H, d]
storage seen as [B, H, L, d]; its tokens are N(0, 1) and the call applies the d^-1/4 of the attention definition.

The theorems leave the signs of B's rows (eigenvectors) free, and rounding decides them: a program that wants the
same outputs from the same inputs orients the rows of what the fit returns (_oriented), and so do the cases.
"""
import functools
import math

import torch

from paper_2302_00787_b200 import binding as fb
from paper_2302_00787_b200 import workloads as wl


def _attn(name, kind, B, H, L, d, M, dtype, variant, causal=False, chunk=0, dv=None, Lk=None, omega="orthogonal",
          layout="bhld", pool="bh", shift=0.0, outliers=0.0, **more):
    c = {"kind": kind, "B": B, "H": H, "L": L, "Lk": L if Lk is None else Lk, "d": d, "dv": d if dv is None else dv, "M": M,
         "dtype": dtype, "variant": variant, "causal": causal, "chunk": chunk, "omega": omega, "layout": layout,
         "pool": pool, "shift": shift, "outliers": outliers, **more}
    return dict(c, name=name) if name else c


def listed():
    return [
        # one small fp32 head, the size of a unit test or of an interactive experiment: latency and launches
        _attn("tiny_f32", "step", 1, 1, 256, 16, 32, "f32", "sderf", omega="iid"),
        # BERT-base encoder layer on a batch of 512-token inputs, SADERF statistics pooled over the batch per head
        _attn("encoder_bf16", "step", 64, 12, 512, 64, 256, "bf16", "saderf", layout="blhd", pool="head"),
        # Conformer-like encoder layer: 8 heads, 4096 frames, heads with a mean of their own
        _attn("bidir_4k_bf16", "step", 8, 8, 4096, 64, 256, "bf16", "sderf", shift=0.1),
        # causal language-model layer, 8192 tokens
        _attn("causal_8k_bf16", "step", 4, 12, 8192, 64, 256, "bf16", "aderf", True, 128),
        # one very long document, wide heads, heavy-tailed tokens
        _attn("long_d128_bf16", "step", 1, 16, 65536, 128, 512, "bf16", "sderf", True, 256, outliers=0.05),
        # a training step of the causal layer
        _attn("train_causal_bf16", "train", 2, 12, 4096, 64, 256, "bf16", "aderf", True, 128, layout="blhd"),
        # fp32 training of a small encoder (ragged length, narrow heads, few features)
        _attn("train_bidir_f32", "train", 4, 8, 1501, 32, 128, "f32", "gerf", omega="iid"),
        # features of a large fp32 batch
        _attn("features_f32", "features", 2, 8, 10007, 64, 256, "f32", "aderf"),
        # kernel classification: Gaussian-kernel scores of 20011 test points from 30000 training points, 16 classes
        _attn("apply_f32", "apply", 1, 1, 20011, 32, 512, "f32", "gerf", dv=16, Lk=30000),
        # one rank of a 65536-token encoder over four ranks
        _attn("slice_bf16", "slice", 1, 16, 16384, 64, 256, "bf16", "sderf", n_ranks=4),
        # a caller with host buffers (inference server without device tensors of its own)
        _attn("host_bf16", "host", 4, 8, 2048, 64, 256, "bf16", "saderf"),
        # the variance study: 2^20 pairs, 32 draws
        {"name": "pairs_f32", "kind": "pairs", "npairs": 2 ** 20, "d": 64, "M": 64, "R": 32, "variant": "aderf"},
    ]


def _logint(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """One more case of the same ranges, at most half of the largest listed case's arithmetic."""
    while True:
        kind = rng.choice(["step"] * 7 + ["train"] * 4 + ["features"] * 2 + ["apply"] * 2 + ["pairs"] * 2 + ["slice"] * 2 + ["host"])
        if kind == "pairs":
            c = {"kind": kind, "npairs": _logint(rng, 1000, 2 ** 20), "d": rng.choice([16, 32, 64, 128]),
                 "M": 16 * rng.randint(1, 16), "R": rng.randint(2, 32), "variant": rng.choice(["aderf", "sderf", "gerf", "posrf"])}
        elif kind in ("slice", "host"):
            c = _attn(None, kind, rng.randint(1, 3), rng.choice([4, 8, 12, 16]), _logint(rng, 500, 8000 if kind == "host" else 24000),
                      64, 256, "bf16", rng.choice(["gerf", "saderf"] if kind == "host" else ["aderf", "sderf", "saderf"]))
            if kind == "slice":
                c.update(n_ranks=rng.randint(2, 8), causal=rng.random() < 0.5)
        else:
            # the tuned head (d = 64, M = 256) half of the time, any other otherwise
            d, M = (64, 256) if rng.random() < 0.5 else (rng.choice([16, 32, 64, 128]), 16 * rng.choice([2, 4, 8, 13, 16, 24, 32]))
            dtype = rng.choice(["bf16", "bf16", "f32"])
            causal = kind in ("step", "train") and rng.random() < 0.5
            chunk = rng.choice([64, 128, 256]) if causal else 0
            L = _logint(rng, 512, 32768)
            if causal:
                L = max(1, L // chunk) * chunk
            c = _attn(None, kind, rng.randint(1, 16), rng.choice([1, 4, 8, 12]), L, d, M, dtype,
                      rng.choice(["gerf", "saderf", "aderf", "sderf"]), causal, chunk,
                      omega=rng.choice(["iid", "orthogonal"]), layout=rng.choice(["bhld", "blhd"]),
                      pool=rng.choice(["bh", "bh", "head"]), outliers=rng.choice([0.0, 0.0, 0.05]))
            if kind == "apply":
                c.update(variant="gerf", dv=rng.choice([16, 32]), Lk=_logint(rng, 512, 32768), layout="bhld", pool="bh", outliers=0.0)
            elif not causal and rng.random() < 0.3:
                c.update(Lk=_logint(rng, 512, 32768))          # cross attention
        if c.get("chunk") and c["B"] * c["H"] * (c["L"] // c["chunk"]) > 65535:
            continue                                                   # the library's limit on (batch, head, chunk)
        if work(c)["flops"] <= 0.5 * work(listed()[-1])["flops"] and _scratch(c) < 20e9:
            return c


def _scratch(c):
    """Bytes of a pass's features, gradients and tensors if all of them were stored."""
    if c["kind"] == "pairs":
        return 4.0 * c["npairs"] * (2 * c["d"] + c["R"])
    return 8.0 * c["B"] * c["H"] * (c["L"] + c["Lk"]) * (c["M"] + c["d"] + c["dv"])


# ---- inputs ----------------------------------------------------------------------------------------------------

@functools.lru_cache(maxsize=None)
def _context():
    """A program keeps one context (its workspace grows to what the largest call needs)."""
    return fb.Context(0)


def _omega(c, seed):
    make = wl.iid_omega if c.get("omega") == "iid" else wl.orthogonal_omega
    return torch.from_numpy(make(c["M"], c["d"], seed % (1 << 31)))


def _tokens(c, gen, L, width, unit):
    """[B, H, L, width] of N(0, 1) entries times `unit`, in the case's layout and type."""
    B, H = c["B"], c["H"]
    shape = (B, L, H, width) if c["layout"] == "blhd" else (B, H, L, width)
    x = torch.randn(shape, generator=gen, device="cuda") * unit
    return x.permute(0, 2, 1, 3) if c["layout"] == "blhd" else x


def _oriented(params, d, variant):
    """The rows of B1 and B2 signed so that B1's row sums are positive (and, where the solver leaves the order of the
    rows free too, ordered by length)."""
    if variant not in ("aderf", "sderf"):
        return params
    B = params[:, d * d:3 * d * d].view(-1, 2, d, d)
    if variant == "aderf" and d == 128:
        order = B[:, 0].norm(dim=2).argsort(dim=1)
        B.copy_(B.gather(2, order[:, None, :, None].expand_as(B)))
    B.mul_(B[:, 0].sum(2).sign()[:, None, :, None])
    return params


def _fitted_before(ctx, Q, K, variant, scale=1.0, per_head=False):
    """Parameters of a program that fits offline, from statistics accumulated in double precision."""
    d, blob = Q.shape[3], []
    for X in (Q, K):
        x = X.double() * scale
        x = x.transpose(0, 1).flatten(1, 2) if per_head else x.flatten(0, 1)
        blob.append((x.transpose(1, 2) @ x / x.shape[1], x.mean(1)))
    (M1, mu4), (M2, mu5) = blob
    stats = torch.cat([M1.flatten(1), M2.flatten(1), mu4, mu5], 1).contiguous()
    return _oriented(ctx.fsharp_fit_params(stats, d, variant), d, variant)


def prepare(case, seed):
    c = case
    gen = torch.Generator(device="cuda").manual_seed(seed)
    ctx = _context()
    if c["kind"] == "pairs":
        n, d = c["npairs"], c["d"]
        X, Y = (torch.rand(n, d, generator=gen, device="cuda") for _ in range(2))
        X, Y = (2.0 * t / t.norm(dim=1, keepdim=True) for t in (X, Y))
        Om = torch.stack([_omega(c, seed * 64 + r) for r in range(c["R"])]).cuda()
        params = _fitted_before(ctx, X[None, None], Y[None, None], c["variant"])
        return {"c": c, "ctx": ctx, "X": X, "Y": Y, "Om": Om, "params": params[0].contiguous()}

    dt = torch.bfloat16 if c["dtype"] == "bf16" else torch.float32
    d, dv, H = c["d"], c["dv"], c["H"]
    unit, scale = (1.0, d ** -0.25) if c["layout"] == "blhd" else (d ** -0.25, 1.0)
    if c["kind"] == "apply":
        unit = 0.5 * d ** -0.5                                        # standardised points times an inverse bandwidth
    Q, K = _tokens(c, gen, c["L"], d, unit), _tokens(c, gen, c["Lk"], d, unit)
    if c["shift"]:
        Q = Q + c["shift"] * torch.randn(1, H, 1, d, generator=gen, device="cuda")
        K = K + c["shift"] * torch.randn(1, H, 1, d, generator=gen, device="cuda")
    if c["outliers"]:
        for X in (Q, K):
            X *= 1.0 + 2.0 * (torch.rand(c["B"], 1, X.shape[2], 1, generator=gen, device="cuda") < c["outliers"])
    if c["kind"] == "apply":                                          # class indicators
        label = torch.randint(dv, (c["B"], H, c["Lk"]), generator=gen, device="cuda")
        V = torch.nn.functional.one_hot(label, dv).float()
    else:
        V = _tokens(c, gen, c["Lk"], dv, 1.0)
    Q, K, V = Q.to(dt), K.to(dt), V.to(dt)
    Om = _omega(c, seed)
    s = {"c": c, "ctx": ctx, "pool": fb.POOL_PER_HEAD if c["pool"] == "head" else fb.POOL_PER_BH, "scale": scale}
    if c["kind"] == "host":
        s.update({k: v.cpu().pin_memory() for k, v in (("Q", Q), ("K", K), ("V", V), ("Om", Om))})
        s["Y"] = torch.empty_like(s["V"] if c["L"] == c["Lk"] else s["Q"]).pin_memory()
        return s
    s.update(Q=Q, K=K, V=V, Om=Om.cuda())
    if c["kind"] == "train":
        s["dY"] = _tokens(c, gen, c["L"], dv, 1.0).to(dt)
    if c["kind"] in ("features", "apply", "slice"):                   # parameters fitted beforehand
        s["params"] = _fitted_before(ctx, Q, K, c["variant"], scale, c["pool"] == "head")
    if c["kind"] == "slice":                                          # what the other ranks have sent
        got = []
        for _ in range(c["n_ranks"] - 1):
            Ko, Vo = _tokens(c, gen, c["Lk"], d, unit).to(dt), _tokens(c, gen, c["Lk"], dv, 1.0).to(dt)
            got.append(ctx.fsharp_attend_key_state(Ko, Vo, s["Om"], s["params"]))
        s["states"], s["shifts"] = torch.cat([g[0] for g in got], 1), torch.cat([g[1] for g in got], 1)
    return s


# ---- one pass ----------------------------------------------------------------------------------------------------

def _fit(s):
    ctx, c = s["ctx"], s["c"]
    stats = ctx.fsharp_stats(s["Q"], s["K"], pool=s["pool"], qk_scale=s["scale"])
    return _oriented(ctx.fsharp_fit_params(stats, c["d"], c["variant"]), c["d"], c["variant"])


def run(state):
    s, c, ctx = state, state["c"], state["ctx"]
    kind = c["kind"]
    if kind == "pairs":
        return ctx.fsharp_pair_estimate(s["X"], s["Y"], s["Om"], s["params"], want_pooled=True)
    if kind == "host":
        return ctx.fsharp_forward_host(s["Q"], s["K"], s["V"], s["Om"], c["variant"], c["causal"], c["chunk"], out=s["Y"])
    at = {"causal": c["causal"], "chunk": c["chunk"], "pool": s["pool"], "qk_scale": s["scale"]}
    if kind == "step":
        return ctx.fsharp_attend(s["Q"], s["K"], s["V"], s["Om"], _fit(s), **at)
    if kind == "train":
        params = _fit(s)
        Y = ctx.fsharp_attend(s["Q"], s["K"], s["V"], s["Om"], params, **at)
        return (Y,) + ctx.fsharp_attend_backward(s["Q"], s["K"], s["V"], s["dY"], s["Om"], params, **at)
    if kind == "features":
        fq = ctx.fsharp_featurize(s["Q"], s["Om"], s["params"], 1, s["pool"], s["scale"], fb.STAB_ROW)
        fk = ctx.fsharp_featurize(s["K"], s["Om"], s["params"], 2, s["pool"], s["scale"], fb.STAB_GROUP)
        return fq + fk
    if kind == "apply":
        return ctx.fsharp_kernel_apply(s["Q"], s["K"], s["V"], s["Om"], s["params"], alpha=-0.5)
    if c["causal"]:       # slice: the handed-on states precede this rank's tokens
        return ctx.fsharp_attend_with_state(s["Q"], s["K"], s["V"], s["Om"], s["params"], s["states"], s["shifts"], causal=True)
    mine, shift = ctx.fsharp_attend_key_state(s["K"], s["V"], s["Om"], s["params"])
    return ctx.fsharp_attend_with_state(s["Q"], None, None, s["Om"], s["params"], torch.cat([s["states"], mine], 1),
                                        torch.cat([s["shifts"], shift], 1))


# ---- what a pass cannot do without, and how exact it is ------------------------------------------------------------

def work(case):
    c = case
    d, M = c["d"], c["M"]
    if c["kind"] == "pairs":
        n, R = c["npairs"], c["R"]
        return {"bytes": 4 * (2 * n * d + R * M * d + R * n) + 8 * n, "flops": 4 * n * R * M * d + 6 * n * d * d}
    U, Lq, Lk, dv = c["B"] * c["H"], c["L"], c["Lk"], c["dv"]
    e = 2 if c["dtype"] == "bf16" else 4
    G = c["H"] if c["pool"] == "head" else U
    quad = 2 * d * d * (Lq + Lk) if c["variant"] == "aderf" else 0         # x^T C x with a dense C
    feat = 2 * M * d * (Lq + Lk) + quad                                    # w^T x
    con = 2 * M * (dv + 1) * (Lq + Lk)                                     # S^T [V | 1], P (S^T [V | 1])
    tri = Lq * c["chunk"] * (M + dv + 1) if c["causal"] and c["chunk"] else 0   # the masked part inside a chunk
    stats = 2 * d * d * (Lq + Lk)
    fit = G * 20 * d ** 3 if c["variant"] in ("aderf", "sderf") else 0
    tensors = U * (Lq + Lk) * (d + dv) * e
    kind = c["kind"]
    if kind == "features":
        return {"bytes": U * (Lq + Lk) * (d * e + 4 * M), "flops": U * feat}
    if kind == "apply":
        return {"bytes": tensors, "flops": U * (feat + con)}
    if kind == "slice":
        return {"bytes": tensors + 4 * U * 65 * 256 * (c["n_ranks"] - 1), "flops": U * (feat + con)}
    flops = U * (stats + feat + con + tri) + fit
    if kind == "train":       # [num | den], R and both dlog products again, dx = dlog W, dV; the inputs once more, the gradients
        flops += U * (2 * feat + 2 * con + con // 2 + 2 * tri)
        tensors += U * (Lq + Lk) * (d + dv) * e + U * Lq * dv * e
    return {"bytes": tensors, "flops": flops}


def tolerance(case):
    c = case
    if c["kind"] == "pairs":
        return {"rel": 3e-5}          # exponents of some tens, in 32 bits
    if c["kind"] == "features" and c["dtype"] == "bf16":
        # fp32 outputs: operands rounded to 11 bits where the kernels of the attention take the shape, to 16 bits for d = 128
        return {"rel": 1e-2 if (c["d"], c["M"]) == (64, 256) else 1e-3 if c["d"] == 128 else 3e-5}
    if c["dtype"] == "bf16":
        return {"rel": 1e-2}
    if c["kind"] in ("features", "apply"):
        return {"rel": 3e-5}
    # refitted in the pass (aderf, sderf): eigenvectors of sample covariances (relative gaps of 1e-3) carry the 32-bit sums of the statistics
    return {"rel": 1e-4 if c["variant"] in ("aderf", "sderf") else 3e-5}
