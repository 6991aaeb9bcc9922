"""The fp32-precision kernels (features, attention, kernel operator, backward pass) at the edges of their tiles: 128 tokens,
feature blocks of 256 (d = 128: 128) in the feature kernels and of 128 in the products, 64 value columns, chunks of 128
tokens whatever the caller's chunk is; against the checker."""
import numpy as np
import pytest
import torch

from oracle import favor_sharp as fs
from tests.gpu_util import TOL, dev, gpu_fit, host, oracle_unit, rel_err
from paper_2302_00787_b200 import binding as fb
from paper_2302_00787_b200 import workloads as wl

pytestmark = pytest.mark.gpu

# (d, dv, M, Lq, Lk, causal, chunk, dtype)
CASES = [
    (16, 16, 16, 1, 300, False, 0, "f32"),          # one query, fewest features
    (32, 128, 48, 127, 129, False, 0, "f32"),       # two tiles of value columns
    (64, 32, 272, 129, 257, False, 0, "bf16"),      # a second feature block of 16
    (64, 64, 1024, 130, 700, False, 0, "f32"),      # most features: row maxima over four blocks
    (128, 16, 144, 260, 140, False, 0, "f32"),      # d = 128: feature blocks of 128
    (16, 64, 208, 64, 64, True, 64, "f32"),         # half a tile
    (32, 32, 128, 192, 192, True, 64, "bf16"),      # the last inner chunk is half full
    (64, 128, 80, 384, 384, True, 128, "f32"),
    (128, 64, 384, 512, 512, True, 256, "bf16"),    # two tiles per chunk
]


def inputs(d, dv, M, Lq, Lk, dtype, seed):
    w = wl.Workload("tiles", 1, 2, Lq, d, dv, M, dtype, "saderf", False, 0, "orthogonal", seed=seed)
    Q, _, V1 = wl.make_qkv(w)
    K, _, V = wl.make_qkv(w.scaled(L=Lk, seed=seed + 1))
    return Q, K, V, V1, wl.make_omega(w)


@pytest.mark.parametrize("d,dv,M,Lq,Lk,causal,chunk,dtype", CASES)
def test_attention_and_gradients_at_tile_edges(d, dv, M, Lq, Lk, causal, chunk, dtype):
    ctx = fb.Context(0)
    Q, K, V, dY, Om = inputs(d, dv, M, Lq, Lk, dtype, 77)
    dQ, dK, dV, ddY, dOm = dev(Q, dtype), dev(K, dtype), dev(V, dtype), dev(dY, dtype), dev(Om)
    _, pr = gpu_fit(ctx, dQ, dK, d, "saderf")
    ctx.set_impl(fb.IMPL_SIMT)
    at = dict(causal=causal, chunk=chunk)
    Y = host(ctx.fsharp_attend(dQ, dK, dV, dOm, pr, **at))
    g = [host(t) for t in ctx.fsharp_attend_backward(dQ, dK, dV, ddY, dOm, pr, **at)]
    assert ctx.status() == 0
    prh = pr.cpu().numpy()
    for h in range(2):
        assert rel_err(Y[0, h], oracle_unit(Q, K, V, Om, prh[h], d, 0, h, causal)) < TOL[dtype]
        ref = fs.favor_sharp_attention_vjp(Q[0, h], K[0, h], V[0, h], dY[0, h], Om, fb.unpack_params(prh[h], d), causal=causal)
        for got, r in zip(g, ref):
            assert rel_err(got[0, h], r) < TOL[dtype]


@pytest.mark.parametrize("d,dv,M,Lq,Lk", [(128, 128, 1024, 3, 5), (16, 16, 16, 1, 1), (32, 128, 1024, 200, 130), (64, 64, 512, 5000, 60)])
def test_sums_start_from_zero_whatever_the_scratch_held(d, dv, M, Lq, Lk):
    """The sums over tokens are cleared by the kernel of the quadratic terms, by more blocks than there are tiles where tiles are few."""
    Q, K, V, dY, Om = inputs(d, dv, M, Lq, Lk, "f32", 5)
    dQ, dK, dV, ddY, dOm = dev(Q), dev(K), dev(V), dev(dY), dev(Om)
    ctx, clean = fb.Context(0), fb.Context(0)
    _, pr = gpu_fit(ctx, dev(inputs(d, dv, M, 600, 600, "f32", 6)[0]), dev(inputs(d, dv, M, 600, 600, "f32", 6)[1]), d, "saderf")
    big = [dev(t) for t in inputs(d, dv, M, 6000, 6000, "f32", 7)[:4]]

    def calls(c):
        return (c.fsharp_attend(dQ, dK, dV, dOm, pr), c.fsharp_kernel_apply(dQ, dK, dV, dOm, pr)) + tuple(
            c.fsharp_attend_backward(dQ, dK, dV, ddY, dOm, pr))

    want = calls(clean)
    for i in range(5):                                    # the scratch full of another call's features before each
        ctx.fsharp_attend_backward(*big, dOm, pr)
        got = calls(ctx)[i]
        assert torch.allclose(got, want[i], rtol=1e-5, atol=1e-5 * float(want[i].abs().max()))
    assert ctx.status() == 0 and clean.status() == 0
    prh = pr.cpu().numpy()
    for h in range(2):
        assert rel_err(host(want[0])[0, h], oracle_unit(Q, K, V, Om, prh[h], d, 0, h, False)) < TOL["f32"]


@pytest.mark.parametrize("d,M,L,dtype", [(16, 16, 1, "f32"), (32, 272, 129, "f32"), (64, 1024, 130, "bf16"), (128, 144, 257, "f32"),
                                         (128, 1024, 128, "bf16")])
@pytest.mark.parametrize("stab", [fb.STAB_NONE, fb.STAB_ROW, fb.STAB_GROUP])
def test_features_at_block_edges(d, M, L, dtype, stab):
    ctx = fb.Context(0)
    Q, K, _, _, Om = inputs(d, 16, M, L, max(L, 4 * d), dtype, 5)
    dQ, dK, dOm = dev(Q, dtype), dev(K, dtype), dev(Om)
    _, pr = gpu_fit(ctx, dQ if L > 1 else dK, dK, d, "saderf")
    ctx.set_impl(fb.IMPL_SIMT)
    phi, ls = ctx.fsharp_featurize(dQ, dOm, pr, 1, stab=stab)
    assert ctx.status() == 0
    for h in range(2):
        p = fb.unpack_params(pr[h], d)
        e = fs.derf_log_features(Q[0, h], Om, p["A"], p["B1"], p["C1"], p["logD"])
        shift = {fb.STAB_NONE: 0.0, fb.STAB_ROW: lambda: host(ls)[0, h][:, None], fb.STAB_GROUP: lambda: host(ls)[0, h]}[stab]
        shift = shift() if callable(shift) else shift
        expect, got = np.exp(e - shift), host(phi)[0, h]
        big = expect > 1e-30
        # an exponent is a sum of d products in fp32: 2^-24 of its largest terms times sqrt(d)
        tol = 2.0 ** -24 * np.abs(e).max() * np.sqrt(d) + 1e-6
        assert np.max(np.abs(got[big] / expect[big] - 1)) < tol
        if stab != fb.STAB_NONE:
            assert got.max() <= 1.0 + 1e-6


@pytest.mark.parametrize("d,M", [(16, 144), (32, 272), (64, 256), (64, 48), (128, 144)])
def test_operands_of_however_many_groups(d, M):
    """W is made one side at a time or both side by side, by the number of groups: a group's features have the same bits."""
    ctx = fb.Context(0)
    gen = torch.Generator(device="cuda").manual_seed(d)
    X = torch.randn(1, 3, 70, d, generator=gen, device="cuda") * d ** -0.25
    Om = dev(wl.orthogonal_omega(M, d, 4))
    _, pr = gpu_fit(ctx, X, X, d, "saderf")
    for side in (1, 2):
        want, _ = ctx.fsharp_featurize(X, Om, pr, side, stab=fb.STAB_ROW)
        for G in (30, 66, 81, 402):
            phi, _ = ctx.fsharp_featurize(X.repeat(1, G // 3, 1, 1), Om, pr.repeat(G // 3, 1), side, stab=fb.STAB_ROW)
            assert torch.equal(phi, want.repeat(1, G // 3, 1, 1))
    assert ctx.status() == 0


def test_unaligned_feature_output_of_the_static_entry_point():
    """phi of fsharp_featurize_static may start on any 4-byte boundary: the result equals the aligned one's."""
    ctx = fb.Context(0)
    Q, K, _, _, Om = inputs(32, 16, 80, 150, 150, "f32", 9)
    dQ, dK, dOm = dev(Q), dev(K), dev(Om)
    _, pr = gpu_fit(ctx, dQ, dK, 32, "saderf")
    out = []
    for off in (0, 1):
        phi = torch.empty(1 * 2 * 150 * 80 + off, device="cuda")[off:].view(1, 2, 150, 80)
        ls = torch.empty(1, 2, 150, device="cuda")
        assert fb.fsharp_featurize_static(dQ, dOm, pr, 1, phi, ls) == 0
        out.append(phi)
    torch.cuda.synchronize()
    assert torch.equal(out[0], out[1])


@pytest.mark.parametrize("d,M,dtype", [(16, 64, "f32"), (64, 256, "f32"), (64, 64, "bf16"), (128, 272, "f32"), (128, 128, "bf16")])
def test_exponents_are_not_biased(d, M, dtype):
    """PosRF features of tokens of 2 sigma (exponents of some tens): the errors of the exponents, regressed on their two parts
    w . x and -|x|^2 / 2, follow neither.  A sum rounded to nearest has errors of either sign; one that is always cut off, or a
    factor log2(e) q^2 that was rounded before it was applied, is off by one unit in the last place or so of the whole: half a unit
    (2^-24) is the bound.  (4000 M errors of 1e-6 determine the slopes to some 1e-3 units.)"""
    gen = torch.Generator(device="cuda").manual_seed(1)
    X = (2.0 * torch.randn(1, 1, 4000, d, generator=gen, device="cuda")).to(torch.bfloat16 if dtype == "bf16" else torch.float32)
    qk = float(np.float32(d ** -0.25))
    Om = dev(wl.orthogonal_omega(M, d, 1))
    I = np.eye(d)
    blob = dev(fb.pack_params({"A": 0 * I, "B1": I, "B2": I, "C1": -0.5 * I, "C2": -0.5 * I, "logD": 0.0}, d)[None])
    ctx = fb.Context(0)
    ctx.set_impl(fb.IMPL_SIMT)
    phi, _ = ctx.fsharp_featurize(X, Om, blob, 1, qk_scale=qk, stab=fb.STAB_NONE)
    assert ctx.status() == 0
    x = qk * X[0, 0].double()
    wx, c = x @ Om.double().T, -0.5 * (x * x).sum(1, keepdim=True)
    e = wx + c - 0.5 * np.log(M)
    ok = (phi[0, 0] > 1e-30) & (phi[0, 0] < 1e30)
    parts = torch.stack([wx[ok], c.expand_as(wx)[ok], torch.ones_like(wx[ok])], 1)
    slope = torch.linalg.lstsq(parts, (phi[0, 0].double().log() - e)[ok][:, None]).solution[:2, 0]
    assert slope.abs().max() < 2.0 ** -24


@pytest.mark.parametrize("d,M,side", [(64, 256, 2), (64, 512, 1), (128, 256, 1), (32, 64, 2)])
def test_no_feature_exceeds_one(d, M, side):
    """Shifts that come from a pass of their own (the group's, and the row's when M needs several feature blocks): the largest
    exponent must not come out above the shift that was taken from it, however far the parts of a sum are from the sum."""
    gen = torch.Generator(device="cuda").manual_seed(2)
    X = 2.0 * torch.randn(8, 4, 500, d, generator=gen, device="cuda")
    qk = d ** -0.25
    ctx = fb.Context(0)
    pr = ctx.fsharp_fit_params(ctx.fsharp_stats(X, X, qk_scale=qk), d, "saderf")
    phi, _ = ctx.fsharp_featurize(X, dev(wl.orthogonal_omega(M, d, 1)), pr, side, qk_scale=qk,
                                  stab=fb.STAB_GROUP if side == 2 else fb.STAB_ROW)
    assert ctx.status() == 0
    top = phi.amax(dim=(2, 3) if side == 2 else 3)
    assert top.max() <= 1.0 and top.min() > 1.0 - 1e-4


@pytest.mark.parametrize("d,causal", [(64, False), (64, True), (128, True)])
def test_sums_over_many_features(d, causal):
    """Outputs and gradients at M = 512, the relative error in the 2-norm.  Sums of 512 terms rounded to nearest err by about
    sqrt(512) / 4 units of 2^-24 (7e-7) in numerator and normaliser; sums that are cut off at every step err by about one unit per
    step, in one direction, and gave 2.3e-6.  Bound 2^-19 (1.9e-6)."""
    ctx = fb.Context(0)
    Q, K, V, dY, Om = inputs(d, d, 512, 1024, 1024, "f32", 31)
    t = [dev(x) for x in (Q, K, V, dY)]
    _, pr = gpu_fit(ctx, t[0], t[1], d, "gerf")
    at = dict(causal=causal, chunk=128)
    got = [host(ctx.fsharp_attend(*t[:3], dev(Om), pr, **at))] + [host(g) for g in ctx.fsharp_attend_backward(*t, dev(Om), pr, **at)]
    assert ctx.status() == 0
    p = fb.unpack_params(pr[0], d)
    ref = (fs.favor_sharp_attention(Q[0, 0], K[0, 0], V[0, 0], Om, p, causal=causal),) + \
        tuple(fs.favor_sharp_attention_vjp(Q[0, 0], K[0, 0], V[0, 0], dY[0, 0], Om, p, causal=causal))
    for g, r in zip(got, ref):
        assert np.linalg.norm(g[0, 0] - r) < 2.0 ** -19 * np.linalg.norm(r)


@pytest.mark.parametrize("level", [40.0, 80.0])
@pytest.mark.parametrize("d,dv", [(32, 16), (16, 128)])
def test_queries_that_see_only_keys_far_below_the_largest(d, dv, level):
    """Causal, fp32: the features of the first 100 keys lie `level` nats below those of the later ones (at 80 nats most of
    what counts lies between 2^-115 and 2^-125, still normal numbers).  What the rows that see nothing else get is as exact as anything, and so are its gradients."""
    rng = np.random.default_rng(8)
    L, M = 256, 48
    Q, K = (0.5 * rng.standard_normal((1, 1, L, d)).astype(np.float32) for _ in range(2))
    V, dY = (rng.standard_normal((1, 1, L, dv)).astype(np.float32) for _ in range(2))
    Om = rng.standard_normal((M, d)).astype(np.float32)
    Q[..., 1], K[..., 1], Om[:, 1] = 0.0, 0.0, 1.0
    K[0, 0, 100:, 1] = level
    dY[0, 0, 100:] = 0.0
    I = np.eye(d)
    p = {"A": 0 * I, "B1": I, "B2": I, "C1": 0 * I, "C2": 0 * I, "logD": 0.0}
    ctx = fb.Context(0)
    t = [dev(x) for x in (Q, K, V, dY)]
    blob = dev(fb.pack_params(p, d)[None])
    at = dict(causal=True, chunk=64)
    Y = host(ctx.fsharp_attend(*t[:3], dev(Om), blob, **at))[0, 0]
    grads = [host(g)[0, 0] for g in ctx.fsharp_attend_backward(*t, dev(Om), blob, **at)]
    assert ctx.status() == 0
    ref = fs.favor_sharp_attention(Q[0, 0], K[0, 0], V[0, 0], Om, p, causal=True)
    # an exponent of 90 nats is known to two units in its last place, 1.5e-5
    assert rel_err(Y[:100], ref[:100]) < 3e-5 and rel_err(Y[100:], ref[100:]) < 3e-5
    for g, r in zip(grads, fs.favor_sharp_attention_vjp(Q[0, 0], K[0, 0], V[0, 0], dY[0, 0], Om, p, causal=True)):
        assert rel_err(g[:100], r[:100]) < 3e-5


@pytest.mark.parametrize("d,M", [(64, 256), (32, 512)])
def test_subnormal_features(d, M):
    """Features below 2^-126 of the row's largest are what fp32 has there: off by half of 2^-149, and the exponent's own error."""
    gen = torch.Generator(device="cuda").manual_seed(2)
    X = 4.0 * torch.randn(1, 1, 2000, d, generator=gen, device="cuda")
    qk = float(np.float32(d ** -0.25))
    Om = dev(wl.orthogonal_omega(M, d, 1))
    I = np.eye(d)
    blob = dev(fb.pack_params({"A": 0 * I, "B1": 2 * I, "B2": I, "C1": -0.5 * I, "C2": -0.5 * I, "logD": 0.0}, d)[None])
    ctx = fb.Context(0)
    phi, ls = ctx.fsharp_featurize(X, Om, blob, 1, qk_scale=qk, stab=fb.STAB_ROW)
    assert ctx.status() == 0
    x = qk * X[0, 0].double()
    e = 2.0 * (x @ Om.double().T) - 0.5 * (x * x).sum(1, keepdim=True) - 0.5 * np.log(M)
    want = (e - ls[0, 0].double()[:, None]).exp()
    tiny = (want < 2.0 ** -126) & (want > 2.0 ** -148)
    assert tiny.sum() > 100
    assert ((phi[0, 0].double() - want).abs() <= 2.0 ** -149 + 1e-4 * want)[tiny].all()


def test_kernel_operator_near_the_smallest_numbers():
    """Shifts of both sides that together are 85 nats below zero (exp: 1e-37) times sums of some thousands: the outputs are normal
    numbers, and the largest of them come out like any other."""
    rng = np.random.default_rng(8)
    d, M = 32, 64
    X, Y = (0.5 * rng.standard_normal((1, 1, L, d)).astype(np.float32) for L in (100, 300))
    Om = rng.standard_normal((M, d)).astype(np.float32)
    I = np.eye(d)
    p = {"A": 0 * I, "B1": I, "B2": I, "C1": -0.5 * I, "C2": -0.5 * I, "logD": 0.0}
    logs = [fs.derf_log_features(x[0, 0], Om, p["A"], I, p["C1"], 0.0) for x in (X, Y)]
    top = logs[0].max() + logs[1].max()
    p["logD"] = 0.5 * (-85.0 - top)
    ctx = fb.Context(0)
    C = np.ones((1, 1, 300, 16), dtype=np.float32)
    out = host(ctx.fsharp_kernel_apply(dev(X), dev(Y), dev(C), dev(Om), dev(fb.pack_params(p, d)[None])))
    assert ctx.status() == 0
    assert rel_err(out[0, 0], fs.kernel_apply(X[0, 0], Y[0, 0], C[0, 0], Om, p, 0.0)) < TOL["f32"]


@pytest.mark.parametrize("d", [16, 32, 64, 128])
@pytest.mark.parametrize("B,H,Lq,Lk,pool", [(1, 1, 1, 1, fb.POOL_PER_BH), (1, 3, 33, 5000, fb.POOL_PER_BH), (2, 19, 129, 700, fb.POOL_PER_HEAD),
                                            (1, 75, 1024, 300, fb.POOL_PER_BH), (1, 2, 9000, 9000, fb.POOL_PER_BH)])
def test_statistics_however_the_tokens_are_cut(B, H, Lq, Lk, pool, d):
    """fp32 tensors: slices of both sides' tokens by lengths and numbers of (batch, head)s; against fp64 sums."""
    ctx = fb.Context(0)
    gen = torch.Generator(device="cuda").manual_seed(d + Lq)
    Q, K = (torch.randn(B, H, L, d, generator=gen, device="cuda") + 0.3 for L in (Lq, Lk))
    st = ctx.fsharp_stats(Q, K, pool=pool)
    assert ctx.status() == 0
    for X, at, mu in ((Q, 0, 2 * d * d), (K, d * d, 2 * d * d + d)):
        x = X.double()
        x = x.transpose(0, 1).flatten(1, 2) if pool == fb.POOL_PER_HEAD else x.flatten(0, 1)
        M, m = x.transpose(1, 2) @ x / x.shape[1], x.mean(1)
        scale = M.diagonal(dim1=1, dim2=2).sqrt()
        # at most 64 products are added in fp32: 64 roundings of sums that are at most the root of the two diagonals' product
        tol = 64 * 2.0 ** -24
        assert ((st[:, at:at + d * d].view(-1, d, d) - M).abs() <= tol * scale[:, :, None] * scale[:, None]).all()
        assert ((st[:, mu:mu + d] - m).abs() <= tol * scale).all()
