"""The bidirectional tensor-core kernels walk one list of 128-token tiles over all (batch, head) units: a unit may lie within
one block, be cut by the end of a block's range, or be spread over every block.  Against the checker at the units where the
ranges end."""
import numpy as np
import pytest
import torch

from oracle import favor_sharp as fs
from tests.gpu_util import TOL, dev, gpu_fit, host, rel_err
from paper_2302_00787_b200 import binding as fb
from paper_2302_00787_b200 import workloads as wl

pytestmark = pytest.mark.gpu

D, M = 64, 256

# (B, H, Lq, Lk, pool)
CASES = [
    (1, 1, 1, 1, fb.POOL_PER_BH),                # one tile, one block
    (1, 1, 100, 20000, fb.POOL_PER_BH),          # one unit over 148 blocks and more tiles than blocks
    (1, 1, 20000, 100, fb.POOL_PER_BH),          # ... on the query side; a unit that nothing cuts
    (1, 3, 300, 6400, fb.POOL_PER_HEAD),         # 150 tiles: blocks of one and two, cut within and at the ends of units
    (50, 6, 128, 128, fb.POOL_PER_HEAD),         # units of one tile, several per block: nothing is cut
    (20, 15, 129, 385, fb.POOL_PER_BH),          # units of two (queries) and four tiles (keys), the last one of one token
    (33, 9, 257, 130, fb.POOL_PER_HEAD),         # W changes within a block, head by head
]


def tensors(B, H, Lq, Lk, spread):
    w = wl.Workload("stream", B, H, Lq, D, D, M, "bf16", "saderf", False, 0, "orthogonal", seed=5)
    Q, _, _ = wl.make_qkv(w)
    K, _, V = wl.make_qkv(w.scaled(L=Lk, seed=6))
    # the size of the keys differs from tile to tile: running maxima that rise within a piece, pieces with unlike shifts
    K = K * (1.0 + spread * np.sin(np.arange(Lk) // 128 * 1.7))[None, None, :, None]
    tq = [dev(x, "bf16") for x in (Q, K, V)]
    Om = wl.make_omega(w)
    return [host(x) for x in tq] + [Om], tq + [dev(Om)]


def checked_units(U, tiles):
    """The first and the last unit, and the units around the ends of some blocks' ranges."""
    n = min(U * tiles, 148)
    ends = [U * tiles * i // n // tiles for i in (1, n // 3, n // 2, n - 1)]
    return sorted({0, U - 1} | {min(max(u, 0), U - 1) for e in ends for u in (e - 1, e)})


@pytest.mark.parametrize("B,H,Lq,Lk,pool", CASES)
def test_units_across_blocks(B, H, Lq, Lk, pool):
    ctx = fb.Context(0)
    (Q, K, V, Om), (dQ, dK, dV, dOm) = tensors(B, H, Lq, Lk, 0.5)
    _, pr = gpu_fit(ctx, dQ, dK, D, "saderf", pool)
    Y = host(ctx.fsharp_attend(dQ, dK, dV, dOm, pr, pool=pool))
    assert ctx.status() == 0
    prh = pr.cpu().numpy()
    for u in sorted(set(checked_units(B * H, -(-Lk // 128))) | set(checked_units(B * H, -(-Lq // 128)))):
        b, h = divmod(u, H)
        ref = fs.favor_sharp_attention(Q[b, h], K[b, h], V[b, h], Om, fb.unpack_params(prh[u if pool == fb.POOL_PER_BH else h], D))
        assert rel_err(Y[b, h], ref) < TOL["bf16"], (b, h)


@pytest.mark.parametrize("copies", [1, 2, 3, 7])
def test_number_of_handed_on_states(copies):
    """Key states of one range of keys, given `copies` times over (1 .. many pieces per merged unit): every feature sum and
    every denominator is multiplied by the same number, so the outputs are those of the range alone."""
    ctx = fb.Context(0)
    (Q, K, V, Om), (dQ, dK, dV, dOm) = tensors(1, 2, 200, 300, 0.5)
    _, pr = gpu_fit(ctx, dQ, dK, D, "saderf")
    st, sh = ctx.fsharp_attend_key_state(dK, dV, dOm, pr)
    Y = host(ctx.fsharp_attend_with_state(dQ, None, None, dOm, pr, torch.cat([st] * copies, 1), torch.cat([sh] * copies, 1)))
    assert ctx.status() == 0
    prh = pr.cpu().numpy()
    for h in range(2):
        ref = fs.favor_sharp_attention(Q[0, h], K[0, h], V[0, h], Om, fb.unpack_params(prh[h], D))
        assert rel_err(Y[0, h], ref) < TOL["bf16"]


@pytest.mark.parametrize("H", [1, 148])           # a unit cut between two blocks; units that one block has all of
@pytest.mark.parametrize("case", ["remnant", "zero"])
def test_feature_whose_column_of_the_state_all_but_vanishes(H, case):
    """Feature 5 (whose exponentials flush to zero in both kernels) is seen by the first 128 keys only (remnant: 2^-13 of the others there, and every other feature then grows by 83
    nats = 2^120) or by no key at all in fp32 (zero); queries may prefer it.  What it contributes is nothing either way, and the
    outputs are those of the other features."""
    K = np.zeros((1, H, 256, D))
    K[..., 0] = 8.0
    K[..., 1] = 83.0
    if case == "remnant":
        K[:, :, :128, 0], K[:, :, :128, 1] = 1.0, 0.0
    rng = np.random.default_rng(4)
    K[..., 2:] = rng.choice([-0.25, 0.0, 0.25], K[..., 2:].shape)
    Q = np.zeros((1, H, 100, D))
    Q[..., 2:] = rng.choice([-0.25, 0.0, 0.25], Q[..., 2:].shape)
    if case == "zero":
        Q[:, :, ::2, 0] = -4.0                   # + 56 nats for feature 5
    V = wl.bf16_round(rng.standard_normal((1, H, 256, D)))
    Om = np.zeros((M, D), dtype=np.float32)
    Om[:, 1] = 1.0
    Om[:, 2:] = rng.choice([-0.5, 0.5], (M, D - 2))
    Om[5] = 0.0
    Om[5, :2] = -14.0, 1.0
    I = np.eye(D)
    p = {"A": 0 * I, "B1": I, "B2": I, "C1": 0 * I, "C2": 0 * I, "logD": 0.0}
    ctx = fb.Context(0)
    pr = dev(np.stack([fb.pack_params(p, D)] * H))
    Y = host(ctx.fsharp_attend(dev(Q, "bf16"), dev(K, "bf16"), dev(V, "bf16"), dev(Om), pr))
    assert ctx.status() == 0
    for h in sorted({0, H // 2, H - 1}):
        assert rel_err(Y[0, h], fs.favor_sharp_attention(Q[0, h], K[0, h], V[0, h], Om, p)) < TOL["bf16"]


# (B, H, Lq, Lk, d, pool)
STATS_CASES = [
    (1, 1, 1, 1, 64, fb.POOL_PER_HEAD),          # one token
    (40, 3, 129, 300, 64, fb.POOL_PER_HEAD),     # ranges that begin and end within sequences; a last tile of one token
    (7, 50, 128, 127, 64, fb.POOL_PER_HEAD),     # one tile per sequence, more groups than ranges
    (9, 2, 257, 128, 128, fb.POOL_PER_HEAD),     # d = 128
    (1, 1, 3, 40000, 128, fb.POOL_PER_BH),       # one group over all SMs
    (2, 2, 20000, 130, 64, fb.POOL_PER_BH),      # sides of unlike length: blocks without a tile
]


@pytest.mark.parametrize("B,H,Lq,Lk,d,pool", STATS_CASES)
def test_statistics_over_a_stream_of_tiles(B, H, Lq, Lk, d, pool):
    """Products of bf16 values are exact in fp32; sums of 256 tokens are rounded to fp32 (256 additions: at most 2^-16 of the sum
    of the magnitudes, here about the diagonal entry), everything after that is fp64."""
    ctx = fb.Context(0)
    gen = torch.Generator(device="cuda").manual_seed(3)
    Q, K = (torch.randn(B, H, L, d, generator=gen, device="cuda").add_(0.3).to(torch.bfloat16) for L in (Lq, Lk))
    st = ctx.fsharp_stats(Q, K, pool=pool).cpu()
    assert ctx.status() == 0
    for side, X in enumerate((Q, K)):
        x = X.double().cpu()
        x = x.transpose(0, 1).flatten(1, 2) if pool == fb.POOL_PER_HEAD else x.flatten(0, 1)
        M = x.transpose(1, 2) @ x / x.shape[1]
        mu = x.mean(1)
        got = st[:, side * d * d:(side + 1) * d * d].reshape(-1, d, d)
        gmu = st[:, 2 * d * d + side * d:2 * d * d + (side + 1) * d]
        assert (got - M).abs().max() <= 2.0 ** -16 * M.abs().max()
        assert (gmu - mu).abs().max() <= 2.0 ** -16 * x.abs().mean(1).max()
