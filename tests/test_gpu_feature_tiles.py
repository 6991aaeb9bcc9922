"""The feature kernels where their store tiles of 32 rows and 32 columns are cut short by the end of the tokens or of the features, where a
block walks many tiles, and on every way out (copies of staged tiles, rows stored directly, single values); against the definition in
fp64 on the device."""
import ctypes as C
import math

import pytest
import torch

from tests.gpu_util import dev, gpu_fit
from paper_2302_00787_b200 import binding as fb
from paper_2302_00787_b200 import workloads as wl

pytestmark = pytest.mark.gpu


def log_features(X, Om, blob, side, d):
    dd, x, w = d * d, X.double(), Om.double()
    A, B, C = (blob[i * dd:(i + 1) * dd].view(d, d) for i in (0, side, 2 + side))
    return (w @ A * w).sum(1) + x @ (w @ B).T + ((x @ C) * x).sum(-1, keepdim=True) + blob[5 * dd] - 0.5 * math.log(Om.shape[0])


@pytest.mark.parametrize("d,M,L,dtype", [(64, 144, 257, "f32"), (32, 208, 33, "bf16"), (16, 240, 300, "f32"), (64, 128, 129, "bf16"),
                                         (64, 256, 12000, "f32"), (32, 256, 31, "f32")])
@pytest.mark.parametrize("stab", [fb.STAB_NONE, fb.STAB_ROW, fb.STAB_GROUP])
def test_features_at_store_tile_edges(d, M, L, dtype, stab):
    ctx = fb.Context(0)
    ctx.set_impl(fb.IMPL_SIMT)
    gen = torch.Generator(device="cuda").manual_seed(M + L)
    X = torch.randn(1, 3, L, d, generator=gen, device="cuda").to(torch.bfloat16 if dtype == "bf16" else torch.float32) * d ** -0.25
    Om = dev(wl.orthogonal_omega(M, d, 4))
    _, pr = gpu_fit(ctx, X, X, d, "saderf")
    phi, ls = ctx.fsharp_featurize(X, Om, pr, 2, stab=stab)
    assert ctx.status() == 0
    check(phi, ls, X, Om, pr, d, stab)


def check(phi, ls, X, Om, pr, d, stab):
    for h in range(3):
        e = log_features(X[0, h], Om, pr[h], 2, d)
        top = {fb.STAB_NONE: torch.zeros(1, device="cuda"), fb.STAB_ROW: e.amax(1, keepdim=True), fb.STAB_GROUP: e.max()}[stab]
        # an exponent is a sum of d products in fp32: 2^-24 of its largest terms times sqrt(d)
        tol = 2.0 ** -24 * float(e.abs().max()) * math.sqrt(d) + 1e-6
        if stab != fb.STAB_NONE:
            assert (ls[0, h].double().view(-1) - top.view(-1)).abs().max() < tol * max(1.0, float(top.abs().max()))
            e = e - ls[0, h].double().view(-1, 1) if stab == fb.STAB_ROW else e - ls[0, h].double()
        big = e > -69.0
        assert (phi[0, h].double() / e.exp() - 1)[big].abs().max() < tol


@pytest.mark.parametrize("d,M,L,dtype", [(64, 144, 257, "f32"), (32, 208, 33, "bf16"), (16, 48, 130, "f32"), (128, 272, 33, "f32"), (128, 144, 257, "f32"),
                                         (128, 272, 257, "bf16"), (128, 144, 33, "bf16"), (64, 80, 38300, "f32"), (64, 96, 12700, "f32"), (128, 144, 12700, "f32"), (128, 144, 25300, "bf16"), (16, 16, 300, "f32")])
@pytest.mark.parametrize("stab", [fb.STAB_ROW, fb.STAB_GROUP])
@pytest.mark.parametrize("past", [0, 1, 4])
def test_features_on_every_way_out(d, M, L, dtype, stab, past):
    """phi `past` words past a 32-byte boundary: on one, rows are stored directly while a block has few tiles and leave as copies beyond
    that (the sizes of 12700 tokens and more); 16 bytes past one always as copies; 4 bytes past one word by word.  Nothing around phi is touched."""
    ctx = fb.Context(0)
    ctx.set_impl(fb.IMPL_SIMT)
    gen = torch.Generator(device="cuda").manual_seed(M + L)
    X = torch.randn(1, 3, L, d, generator=gen, device="cuda").to(torch.bfloat16 if dtype == "bf16" else torch.float32) * d ** -0.25
    Om = dev(wl.orthogonal_omega(M, d, 4))
    _, pr = gpu_fit(ctx, X, X, d, "saderf")
    guard = 64
    buf = torch.full((past + guard + 3 * L * M + guard,), -7.0, device="cuda")
    assert buf.data_ptr() % 256 == 0
    phi = buf[past + guard:past + guard + 3 * L * M].view(1, 3, L, M)
    ls = torch.empty((1, 3, L) if stab == fb.STAB_ROW else (1, 3), device="cuda")
    dims = fb.make_dims(1, 3, L, L, d, d, M, q=X, k=X)
    assert ctx.lib.fsharp_featurize(ctx._h, X.data_ptr(), Om.data_ptr(), pr.data_ptr(), 2, C.byref(dims), fb._dtype_code(X), 1.0, stab,
                                    phi.data_ptr(), ls.data_ptr()) == 0
    assert ctx.status() == 0
    check(phi, ls, X, Om, pr, d, stab)
    assert bool((buf[:past + guard] == -7.0).all()) and bool((buf[past + guard + 3 * L * M:] == -7.0).all())


@pytest.mark.parametrize("d,M,groups,dtype", [(16, 144, 3, "f32"), (32, 272, 3, "f32"), (64, 256, 3, "f32"), (64, 48, 90, "f32"), (128, 144, 3, "f32"),
                                              (64, 256, 3, "bf16"), (64, 256, 90, "bf16")])
def test_features_of_a_dense_quadratic_form(d, M, groups, dtype):
    """All fits give a diagonal A; a blob may hold any.  bf16: the operand images of the tensor-core kernels."""
    ctx = fb.Context(0)
    gen = torch.Generator(device="cuda").manual_seed(d + M)
    X = torch.randn(1, 3, 150, d, generator=gen, device="cuda").to(torch.bfloat16 if dtype == "bf16" else torch.float32) * d ** -0.25
    Om = dev(wl.orthogonal_omega(M, d, 4))
    _, pr = gpu_fit(ctx, X, X, d, "saderf")
    S = torch.randn(3, d, d, generator=gen, device="cuda", dtype=torch.float64) * 0.02 / d ** 0.5
    pr[:, :d * d] += (S + S.transpose(1, 2)).flatten(1)
    n = groups // 3
    for side in (1, 2):
        phi, ls = ctx.fsharp_featurize(X.repeat(1, n, 1, 1), Om, pr.repeat(n, 1), side, stab=fb.STAB_ROW)
        assert ctx.status() == 0 and torch.equal(phi, phi[:, :3].repeat(1, n, 1, 1))
        for h in range(3):
            e = log_features(X[0, h], Om, pr[h], side, d)
            w, A = Om.double().abs(), pr[h, :d * d].view(d, d).abs()
            # as above, and the same of the terms of w^T A w; tensor-core kernels: W rounded to 11 bits (the bound of their other tests)
            tol = 2.0 ** -24 * float(e.abs().max() + (w @ A * w).sum(1).max()) * math.sqrt(d) + 1e-6 if dtype == "f32" else 1e-2
            assert (ls[0, h].double() - e.amax(1)).abs().max() < tol * max(1.0, float(e.abs().max()))
            assert (phi[0, h].double() - (e - ls[0, h].double()[:, None]).exp()).abs().max() < tol
