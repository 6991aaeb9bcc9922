"""The feature kernels where their store tiles of 32 rows and 32 columns are cut short by the end of the tokens or of the features, and
where a block walks many tiles; against the definition in fp64 on the device."""
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
