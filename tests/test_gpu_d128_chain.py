"""The chain of kernels for bf16, d = dv = 128, causal (feature maps, running key-side sums, query side) where its work is cut
differently: one tile, one chunk, one segment for want of SMs, as many segments as chunks, segments whose totals are added up in
pieces, one, two (whole and half) and three blocks of features; against the fp32 kernels on the same numbers."""
import numpy as np
import pytest
import torch

from tests.gpu_util import dev, gpu_fit, host
from paper_2302_00787_b200 import binding as fb
from paper_2302_00787_b200 import workloads as wl

pytestmark = pytest.mark.gpu


def row_bound(ctx, Q, K, V, Om, pr, at):
    """What the chain's roundings may move every output value by, against the fp32 tensors' result.  Numerator and denominator are sums
    whose terms carry three roundings to bf16 each (phi(Q); phi(K); the score or the running sum), the quotient one more: to first
    order 7 x 2^-9 of the attention applied to |V|.  Second order and the exponents from two parts of W (16 bits): one more."""
    return 8 * 2.0 ** -9 * host(ctx.fsharp_attend(Q.float(), K.float(), V.float().abs(), Om, pr, **at))


@pytest.mark.parametrize("B,H,L,M,chunk,variant", [
    (1, 1, 128, 128, 128, "sderf"),       # one tile
    (1, 1, 256, 256, 256, "aderf"),       # one chunk of two tiles: nothing precedes it; a dense C
    (2, 19, 384, 512, 128, "saderf"),     # 152 (batch, head, feature block)s: one segment each
    (1, 3, 5120, 128, 256, "sderf"),      # a segment per chunk
    (1, 16, 1024, 512, 128, "sderf"),     # two segments of four chunks, the first added up in two pieces
    (1, 5, 2816, 384, 256, "aderf"),      # a last segment of one chunk; the second block of features half full
    (1, 2, 512, 640, 256, "sderf"),       # three blocks of features: row maxima by a pass of their own
])
def test_chain_against_fp32_kernels(B, H, L, M, chunk, variant):
    ctx = fb.Context(0)
    w = wl.Workload("chain", B, H, L, 128, 128, M, "bf16", variant, True, chunk, "orthogonal", outlier_frac=0.05, seed=9)
    Q, K, V = (dev(t, "bf16") for t in wl.make_qkv(w))
    Om = dev(wl.make_omega(w))
    _, pr = gpu_fit(ctx, Q, K, 128, "saderf" if L < 512 else variant)
    at = dict(causal=True, chunk=chunk)
    Y = host(ctx.fsharp_attend(Q, K, V, Om, pr, **at))
    assert torch.equal(ctx.fsharp_attend(Q, K, V, Om, pr, **at).float().cpu().double(), torch.from_numpy(Y))
    ref = host(ctx.fsharp_attend(Q.float(), K.float(), V.float(), Om, pr, **at))
    assert ctx.status() == 0
    assert (np.abs(Y - ref) <= row_bound(ctx, Q, K, V, Om, pr, at)).all()
    # the first token sees itself alone
    assert np.abs(Y[:, :, 0] - host(V)[:, :, 0]).max() < 1e-2 * np.abs(host(V)[:, :, 0]).max()


@pytest.mark.parametrize("M,variant", [(512, "sderf"), (384, "aderf"), (256, "sderf"), (512, "mixed"), (256, "mixed")])
def test_blocks_over_many_tiles(M, variant):
    """16 (batch, head)s of 40 token tiles.  Two blocks of features: a pair of blocks exchanges its rows' maxima over eight or nine
    tiles, four or five per warpgroup, so that every place and barrier of the exchange is used again.  C = gamma I: the epilogue's reads
    of a tile are done before the next one is copied over it.  mixed: groups with C = gamma I between groups with a dense C.  Always the
    same bits."""
    ctx = fb.Context(0)
    w = wl.Workload("chain", 2, 8, 5120, 128, 128, M, "bf16", "sderf", True, 256, "orthogonal", outlier_frac=0.05, seed=3)
    Q, K, V = (dev(t, "bf16") for t in wl.make_qkv(w))
    Om = dev(wl.make_omega(w))
    st, pr = gpu_fit(ctx, Q, K, 128, "sderf" if variant == "mixed" else variant)
    if variant == "mixed":
        pr[1::3] = ctx.fsharp_fit_params(st, 128, "aderf")[1::3]
    at = dict(causal=True, chunk=256)
    Y = ctx.fsharp_attend(Q, K, V, Om, pr, **at)
    ref = host(ctx.fsharp_attend(Q.float(), K.float(), V.float(), Om, pr, **at))
    assert (np.abs(host(Y) - ref) <= row_bound(ctx, Q, K, V, Om, pr, at)).all()
    for _ in range(100):
        assert torch.equal(ctx.fsharp_attend(Q, K, V, Om, pr, **at), Y)
    assert ctx.status() == 0
