"""Calls from several host threads, each with a context and a stream of its own: same kernels, launched at the same time with
unlike amounts of shared memory."""
import threading

import numpy as np
import pytest
import torch

from paper_2302_00787_b200 import binding as fb
from paper_2302_00787_b200 import workloads as wl

pytestmark = pytest.mark.gpu


def fits(d, G, variant):
    rng = np.random.default_rng(d)
    X = rng.standard_normal((8 * d, d)) / d ** 0.5
    M1 = X.T @ X / 8 + 0.1 * np.eye(d)
    blob = torch.from_numpy(np.tile(np.concatenate([M1.ravel(), M1.ravel(), np.zeros(2 * d)]), (G, 1))).cuda()
    return lambda ctx, out: ctx.fsharp_fit_params(blob, d, variant, out=out), torch.empty(G, fb.params_doubles(d), dtype=torch.float64, device="cuda")


def pairs(d, M, R):
    X = torch.full((300, d), 0.1, device="cuda")
    Om = torch.stack([torch.from_numpy(wl.orthogonal_omega(M, d, r)) for r in range(R)]).cuda()
    I = np.eye(d)
    blob = torch.from_numpy(fb.pack_params({"A": 0 * I, "B1": I, "B2": I, "C1": -0.5 * I, "C2": -0.5 * I, "logD": 0.0}, d)).cuda()
    return lambda ctx, out: ctx.fsharp_pair_estimate(X, X, Om, blob, want_variance=False, est=out), torch.empty(R, 300, device="cuda")


@pytest.mark.parametrize("jobs", [[("fits", 64, 1, "sderf"), ("fits", 64, 700, "sderf"), ("fits", 64, 200, "aderf")],
                                  [("fits", 16, 1, "aderf"), ("fits", 64, 1, "gerf"), ("fits", 32, 1, "gerf")],
                                  [("pairs", 64, 16, 1), ("pairs", 64, 128, 2), ("pairs", 64, 48, 3)]])
def test_launches_of_one_kernel_from_several_threads(jobs):
    work = [{"fits": fits, "pairs": pairs}[j[0]](*j[1:]) for j in jobs]
    want = []
    for call, out in work:
        call(fb.Context(0), out)
        torch.cuda.synchronize()
        want.append(out.clone())
    ctxs = [fb.Context(0, stream=torch.cuda.Stream()) for _ in work]
    failed = []

    def run(i):
        try:
            for _ in range(1500):
                work[i][0](ctxs[i], work[i][1])
        except fb.FsharpError as e:
            failed.append((jobs[i], e.code))

    threads = [threading.Thread(target=run, args=(i,)) for i in range(len(work))]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    torch.cuda.synchronize()
    assert not failed
    for (_, out), w, c in zip(work, want, ctxs):
        assert c.status() == 0 and torch.equal(out, w)
