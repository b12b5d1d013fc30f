"""FP64 solves through the fixed-point block kernels at their edges.

Widths at and beside the kernels' buckets (4, 8, 12 and, beyond the
fixed-point range, 13), right-hand sides of very different scales (every
column of the coefficients has its own exponent) and a dependent column.  An
FP64 solve's true residual is recomputed by the library in FP64; here the
oracle recomputes it for every pair, and every pair has to meet 10 tol, as in
the other solve tests.
"""
import numpy as np
import pytest
import torch

from oracle import wilson as W
from paper_1205_0359_gb300 import dsbcg, synth

pytestmark = pytest.mark.gpu
DEV = torch.device("cuda")
TOL = 1e-11


def _solve(dims, m, s, scale, dependent):
    rng = np.random.Generator(np.random.PCG64(100 + m))
    U = synth.su3_links(dims, 0.4, rng)
    n = 12 * synth.volume(dims)
    B = synth.gaussian_rhs(n, m, rng) * (scale ** np.arange(m))[:, None]
    if dependent:
        B[m - 1] = B[0] - B[1]
    sigma = synth.log_shifts(1e-2, 1.0, s)
    ctx = dsbcg.Context(dims, torch.from_numpy(U).to(DEV), 0.12)
    X, st = ctx.solve(torch.from_numpy(B).to(DEV), sigma, TOL, storage="fp64")
    ctx.close()
    assert st["code"] == 0 and st["true_relres"].max() <= TOL
    X = X.cpu().numpy()
    for j in range(s):
        R = B - sigma[j] * X[j] - W.A_vec(U, 0.12, dims, X[j])
        assert (np.linalg.norm(R, axis=1) <= 10 * TOL * np.linalg.norm(B, axis=1)).all(), j
    return st


@pytest.mark.parametrize("m", [1, 3, 4, 5, 8, 9, 12, 13])
def test_widths_around_the_buckets(m):
    _solve((4, 4, 2, 5), m, 3, 1.0, False)


@pytest.mark.parametrize("m,scale", [(4, 1e-9), (6, 1e5), (12, 1e-3)])
def test_right_hand_sides_of_different_scales(m, scale):
    _solve((4, 4, 4, 4), m, 2, scale, False)


@pytest.mark.parametrize("m", [4, 11])
def test_dependent_column_deflates(m):
    assert _solve((4, 4, 4, 4), m, 2, 1.0, True)["deflations"] >= 1
