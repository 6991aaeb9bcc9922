"""Pair estimates and closed-form variances at the edges of the kernels' tiles (128 pairs, column tiles of whole draws or
of pieces of one draw, d = 16 .. 128, rows that do not start on 16-byte boundaries) against the checker."""
import numpy as np
import pytest
import torch

from oracle import favor_sharp as fs
from tests.gpu_util import dev, host
from paper_2302_00787_b200 import binding as fb
from paper_2302_00787_b200 import workloads as wl

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("d,M,R,npairs,variant,offset", [
    (16, 16, 1, 1, "gerf", 0),             # smallest
    (16, 48, 7, 129, "sderf", 1),          # draws do not fill the last column tile; unaligned rows
    (32, 208, 5, 300, "aderf", 0),         # one draw over two column tiles, padded
    (64, 64, 3, 127, "aderf", 3),          # odd number of units
    (64, 1024, 2, 130, "posrf", 0),        # most features
    (128, 112, 4, 257, "aderf", 0),        # d = 128: operands streamed twice
    (128, 256, 1, 128, "gerf", 2),
])
def test_pair_kernels_at_tile_edges(d, M, R, npairs, variant, offset):
    ctx = fb.Context(0)
    X, Y = wl.make_pairs(max(npairs, 4 * d), d)
    dX, dY = dev(X), dev(Y)
    pr = ctx.fsharp_fit_params(ctx.fsharp_stats(dX[None, None], dY[None, None]), d, variant)
    X, Y = X[:npairs], Y[:npairs]
    bX, bY = (torch.empty(npairs * d + offset, device="cuda")[offset:].view(npairs, d) for _ in range(2))
    bX.copy_(dX[:npairs])
    bY.copy_(dY[:npairs])
    Om = np.stack([wl.orthogonal_omega(M, d, 100 + r) for r in range(R)])
    est, var, pooled = ctx.fsharp_pair_estimate(bX, bY, dev(Om), pr, want_pooled=True)
    assert ctx.status() == 0
    p = fb.unpack_params(pr[0], d)
    ref = np.stack([fs.pair_estimate(X, Y, Om[r], p) for r in range(R)])
    # an exponent is a sum of 2 d products (+ 4 terms) of magnitudes up to some tens in fp32: 32 * 2^-24 * sqrt(2 d) <= 3e-5
    assert np.max(np.abs(host(est) - ref) / ref) < 3e-5
    refv = fs.pair_closed_form_variance(X, Y, p, M)
    # fp64 throughout; the difference of two exponentials loses at most their ratio to the result
    k2 = np.exp(2.0 * np.sum(X.astype(np.float64) * Y, axis=1)) / M
    assert np.max(np.abs(host(var) - refv) / (np.abs(refv) + k2)) < 1e-10
    got = host(pooled)
    if R > 1:
        emp, cf = fs.pair_pooled_relative_variance(host(est), X, Y, refv)
        assert abs(got[0] - emp) <= 1e-9 * abs(emp)
    else:                                   # one draw has no sample variance
        cf = float((refv / np.exp(2.0 * np.sum(X.astype(np.float64) * Y, axis=1))).mean())
        assert got[0] == 0.0
    assert abs(got[1] - cf) <= 1e-9 * abs(cf)


@pytest.mark.parametrize("d", [16, 32, 64, 128])
def test_estimates_are_not_biased(d):
    """PosRF estimates of 40000 pairs: the mean of the relative errors.  Rounded to nearest, the sums that make an exponent of some
    ten units have errors of either sign and a mean of 1e-8 (4 x 40000 of them, each below 1e-6); sums that are cut off at every
    step gave 4e-7 to 1.8e-6.  Bound: half a unit in the last place of the exponents' products (8 to 16), 2^-21."""
    gen = torch.Generator(device="cuda").manual_seed(3)
    X, Y = (torch.rand(40000, d, generator=gen, device="cuda") for _ in range(2))
    X, Y = (2.0 * t / t.norm(dim=1, keepdim=True) for t in (X, Y))
    Om = torch.stack([dev(wl.orthogonal_omega(64, d, r)) for r in range(4)])
    I = np.eye(d)
    blob = dev(fb.pack_params({"A": 0 * I, "B1": I, "B2": I, "C1": -0.5 * I, "C2": -0.5 * I, "logD": 0.0}, d))
    ctx = fb.Context(0)
    est, _ = ctx.fsharp_pair_estimate(X, Y, Om, blob, want_variance=False)
    assert ctx.status() == 0
    x, y = X.double(), Y.double()
    e = (x + y) @ Om.double().transpose(1, 2) - 0.5 * ((x * x).sum(1) + (y * y).sum(1))[:, None]
    assert (est.double() / e.exp().mean(2) - 1).mean().abs() < 2.0 ** -21
