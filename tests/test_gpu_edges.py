"""Kernels and dispatch branches at the edges of their tiles, remainders and
ranges, against the oracle on the same inputs."""
import numpy as np
import pytest
import torch

import oracle as orc
from paper_1909_07570_gb300 import inputs, native

pytestmark = pytest.mark.gpu


def _dev(a, dt):
    return torch.tensor(np.asarray(a), dtype=dt, device="cuda")


# FP64: a few sweeps amplify 1e-16 rounding by far less than 1e-9. FP32: sums of at
# most a few thousand positive terms, a few sweeps: 1e-4 (the one-sweep bound of the
# FP32 kernels).
_TOL = {torch.float64: 1e-9, torch.float32: 1e-4}


@pytest.mark.parametrize("dt", [torch.float64, torch.float32])
@pytest.mark.parametrize("jobs", [
    [((1, 1, 1), (1, 1, 1)), ((5, 1, 3), (2, 1, 2))],
    [((4, 4, 4), (5, 5, 5)), ((40, 40, 40), (3, 4, 5)), ((7, 33, 18), (4, 8, 1))],
    [((9, 3, 31), (8, 3, 8)), ((3, 65, 4), (3, 7, 4))],
    [((17, 20, 24), (16, 9, 13)), ((33, 6, 7), (12, 6, 7))],
    [((64, 2, 64), (4, 2, 4))],
    [((120, 4, 120), (4, 4, 4))],      # X x_2 F2^T beyond a block: N2 far below N1 and N3
    [((10, 12, 11), (17, 4, 20))],     # a multirank beyond 16
])
def test_small_batched_edges(dt, jobs):
    probs = [inputs.small_problem(d, 3, m, 2, seed=31 + i) for i, (d, m) in enumerate(jobs)]
    dev = [(_dev(X, dt), [_dev(f, dt) for f in F0], _dev(G0, dt)) for X, _, F0, G0, _ in probs]
    errs = native.ntd_fit_small_batched(dev, 3).cpu().numpy()
    tol = _TOL[dt]
    for (X, _, F0, G0, _), (Xd, F, G), e in zip(probs, dev, errs):
        Xr = Xd.double().cpu().numpy()
        Fo, Go, _ = orc.ntd_fit(Xr, [f.astype(np.float32).astype(float) if dt == torch.float32 else f
                                     for f in F0],
                                G0.astype(np.float32).astype(float) if dt == torch.float32 else G0, 3)
        for a, b in zip(F + [G], Fo + [Go]):
            np.testing.assert_allclose(a.double().cpu().numpy(), b, rtol=tol, atol=tol * 1e-3)
        assert e == pytest.approx(orc.rel_err_tucker(Xr, Go, Fo), abs=tol)
