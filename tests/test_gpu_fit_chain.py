"""The chain of fit kernels for d = 64 and 128 (ADERF, SDERF) where groups of one launch take different ways: ordinary spectra
through the chain, eigenvalues equal to rounding through the Jacobi solver behind it, more groups than SMs."""
import numpy as np
import pytest
import torch

from oracle import favor_sharp as fs
from paper_2302_00787_b200 import binding as fb
from tests.test_gpu_parity import assert_fit_close

pytestmark = pytest.mark.gpu


def matrices(d, kind, rng):
    Qm, _ = np.linalg.qr(rng.standard_normal((d, d)))
    lam = {"plain": rng.uniform(0.1, 0.9, d), "equal": np.full(d, 0.3), "clusters": np.repeat(np.linspace(0.1, 0.5, 8), d // 8),
           "wide": np.geomspace(1e-2, 1e2, d)}[kind]
    M1 = (Qm * lam) @ Qm.T
    return 0.5 * (M1 + M1.T)


@pytest.mark.parametrize("variant", ["sderf", "aderf"])
@pytest.mark.parametrize("d,copies", [(64, 1), (64, 60), (128, 1)])
def test_mixed_groups(variant, d, copies):
    rng = np.random.default_rng(d + copies)
    kinds = ["plain", "equal", "clusters", "wide"]
    blobs, refs = [], []
    for kind in kinds:
        M1 = matrices(d, kind, rng)
        M2 = 0.5 * M1 + 0.1 * np.eye(d)
        mu4, mu5 = 0.01 * rng.standard_normal((2, d)) if kind == "plain" else np.zeros((2, d))
        refs.append(fs.FITS[variant]({"M1": M1, "M2": M2, "mu4": mu4, "mu5": mu5, "mu3": float(mu4 @ mu5) / d, "d": d}))
        blobs.append(np.concatenate([M1.ravel(), M2.ravel(), mu4, mu5]))
    ctx = fb.Context(0)
    pr = ctx.fsharp_fit_params(torch.from_numpy(np.stack(blobs * copies)).cuda(), d, variant)
    assert ctx.status() == 0
    # copies of one matrix get the same bits wherever they run
    first = pr[:len(kinds)]
    assert torch.equal(pr.view(copies, len(kinds), -1), first.expand(copies, -1, -1))
    for g, ref in enumerate(refs):
        # "wide": either side's eigenvalues of Z are exact to 2^-53 |Z| d, that is 2^-53 d cond(Z) of the smallest, which carries
        # the largest entries of B1^T B1; Z has the eigenvalues lam (lam / 2 + 1/10), cond 5e6
        assert_fit_close(fb.unpack_params(first[g], d), ref, d, max(1e-8, 2.0 ** -53 * d * 5e6) if kinds[g] == "wide" else 1e-8)
    # Jacobi sweeps: none in the chain; vectors of eigenvalues that agree to rounding are not orthonormal there, and the Jacobi solver
    # takes over.  (A multiple of the identity goes there too and needs no sweep.)
    sweeps = first[:, 5 * d * d + 3].tolist()
    assert sweeps[0] == 0 and sweeps[kinds.index("clusters")] > 0


@pytest.mark.parametrize("variant", ["sderf", "aderf"])
@pytest.mark.parametrize("d", [64, 128])
def test_statistics_on_any_8_byte_boundary(d, variant):
    """The statistics blob is an array of doubles: one that starts 8 bytes past a 16-byte boundary gives the same bits."""
    rng = np.random.default_rng(d)
    M1, M2 = matrices(d, "plain", rng), matrices(d, "plain", rng)
    blob = torch.from_numpy(np.tile(np.concatenate([M1.ravel(), M2.ravel(), 0.01 * rng.standard_normal(2 * d)]), (3, 1))).cuda()
    ctx = fb.Context(0)
    want = ctx.fsharp_fit_params(blob, d, variant)
    shifted = torch.empty(blob.numel() + 1, dtype=torch.float64, device="cuda")[1:].view_as(blob).copy_(blob)
    assert shifted.data_ptr() % 16 == 8
    assert torch.equal(ctx.fsharp_fit_params(shifted, d, variant), want)
    assert ctx.status() == 0


@pytest.mark.parametrize("variant", ["posrf", "gerf", "saderf"])
@pytest.mark.parametrize("d,G", [(16, 201), (32, 99), (32, 600), (64, 102), (64, 300), (64, 2500), (128, 150), (128, 500), (128, 1200)])
def test_closed_forms_however_many_groups(d, G, variant):
    """The closed forms share a group's rows out to fewer blocks the more groups there are: the same bits as group by group; a
    violated constraint in the last group is reported whichever block finds it."""
    rng = np.random.default_rng(d)
    X = rng.standard_normal((3, 4 * d, d)) / d ** 0.5
    blob = torch.from_numpy(np.stack([np.concatenate([(x.T @ x / 8).ravel(), (x.T @ x / 4).ravel(), 0.1 * x[0], 0.1 * x[1]]) for x in X])).cuda()
    ctx = fb.Context(0)
    want = torch.cat([ctx.fsharp_fit_params(blob[g:g + 1], d, variant) for g in range(3)])
    many = blob.repeat((G + 2) // 3, 1)[:G].contiguous()
    assert torch.equal(ctx.fsharp_fit_params(many, d, variant), want.repeat((G + 2) // 3, 1)[:G])
    assert ctx.status() == 0
    many[G - 1, d * d - 1] = float("nan")                  # (a diagonal entry: SADERF's M1 is no longer positive there)
    ctx.fsharp_fit_params(many, d, variant)
    assert ctx.status() == (-6 if variant == "saderf" else -7)
