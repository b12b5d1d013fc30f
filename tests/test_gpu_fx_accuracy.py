"""Precision and range of the block fixed-point kernels where a true residual
does not repair them.

* The block update, V = W S and shift update of FP64 solves: the iterate after
  five block steps, without any restart, against the block Galerkin iterate of
  Eq. 3.2 from the oracle's fully orthogonalised basis.  A step is four passes
  of up to m products each, so in FP64 arithmetic a column's relative error is
  below 5 x 4 m 2^-53 times the condition number of sigma + A; an FP64 emulation
  of the recurrences on the CPU gives 1e-15 for these fields, coefficients held
  to 44 bits 1e-13 and to 29 bits (one limb) 5e-9.  Right-hand sides: Gaussian,
  and sources that fall by two decades per hop, so that the rows of V and P,
  which share one exponent, hold columns of very different size.
* The 64-bit sums of the stencil at their largest: eight hops whose terms all
  add up and a diagonal term 2^4 above its neighbours (2^62.8 of 2^63).
"""
import numpy as np
import pytest
import torch

from oracle import wilson as W
from oracle.dsbcg import galerkin_iterate
from paper_1205_0359_gb300 import dsbcg, synth

pytestmark = pytest.mark.gpu
DEV = torch.device("cuda")


def _coords(dims):
    return np.array(list(np.ndindex(*dims[::-1])))[:, ::-1]


def _sources(dims, m, rng):
    """Column i falls as 10^-(2 hops) from a site of its own."""
    c, L = _coords(dims), np.array(dims)
    B = synth.gaussian_rhs(12 * len(c), m, rng).reshape(m, len(c), 12)
    for i in range(m):
        d = np.abs(c - c[(5 * i + 3) % len(c)])
        B[i] *= 10.0 ** (-2.0 * np.minimum(d, L - d).sum(1))[:, None]
    return B.reshape(m, -1)


@pytest.mark.parametrize("m", [1, 4, 5, 8, 12, 13])
@pytest.mark.parametrize("kind", ["gaussian", "sources"])
def test_iterate_without_restarts(m, kind):
    dims, kappa, k, sigma = (4, 4, 2, 2), 0.12, 5, [0.5, 2.0]
    rng = np.random.Generator(np.random.PCG64(7 + m))
    U = synth.su3_links(dims, 0.4, rng)
    n = 12 * synth.volume(dims)
    B = synth.gaussian_rhs(n, m, rng) if kind == "gaussian" else _sources(dims, m, rng)
    A = W.dense_A(U, kappa, dims)
    ev = np.linalg.eigvalsh(A)
    ctx = dsbcg.Context(dims, torch.from_numpy(U).to(DEV), kappa)
    X, st = ctx.solve(torch.from_numpy(B).to(DEV), sigma, 0.0, storage="fp64", max_block_steps=k, refine=False,
                      freeze=False, poll_every=1, max_restarts=0, raise_on_error=False)
    ctx.close()
    assert st["code"] == 1 and st["block_steps"] == k and st["restarts"] == 0
    G = galerkin_iterate(A, B, sigma, k)
    err = np.linalg.norm(X.cpu().numpy() - G, axis=-1) / np.linalg.norm(G, axis=-1)
    for j, sg in enumerate(sigma):
        assert err[j].max() <= 5 * 4 * m * 2.0 ** -53 * (sg + ev[-1]) / (sg + ev[0]), j


def _aligned_link(forward):
    """SU(3) with row 0 (column 0 for a backward hop) e^{i pi/4} / sqrt(3) throughout."""
    w = np.exp(2j * np.pi / 3)
    F = np.array([[w ** (i * j) for j in range(3)] for i in range(3)]) / np.sqrt(3)
    F[0] *= np.exp(0.25j * np.pi)
    F[1] /= np.linalg.det(F)
    return F if forward else F.T


@pytest.mark.parametrize("comp", [0, 3, 6, 9])
@pytest.mark.parametrize("dag", [False, True])
def test_largest_sums(comp, dag):
    dims, site = (4, 4, 4, 4), (1, 2, 1, 2)
    kappa = 1.0 - 2.0 ** -20
    V = synth.volume(dims)
    U = synth.su3_links(dims, 0.5, np.random.Generator(np.random.PCG64(6)))
    at = lambda c: c[0] + 4 * (c[1] + 4 * (c[2] + 4 * c[3]))
    flat = U.reshape(V, 4, 3, 3)
    for mu in range(4):
        back = tuple(c - (d == mu) for d, c in enumerate(site))
        flat[at(site), mu] = _aligned_link(True)
        flat[at(back), mu] = _aligned_link(False)
    op, ref, adj = ("Ddag", W.Ddag_vec, W.D_vec) if dag else ("D", W.D_vec, W.Ddag_vec)
    e = np.zeros((1, 12 * V), dtype=complex)
    i = 12 * at(site) + comp
    e[0, i] = 1.0
    row = adj(U, kappa, dims, e).conj()[0]                    # row i of the operator
    row[np.abs(row) < 1e-12] = 0.0
    F = (1.0 - 2.0 ** -52) * (np.sign(row.real) - 1j * np.sign(row.imag))
    F[12 * at(site):12 * at(site) + 12] = 0.0
    F[i] = 16.0 * (1.0 - 2.0 ** -52)
    want = ref(U, kappa, dims, F[None])
    assert want[0, i].real > 2.0 ** 5.78                      # of 2^6: a unit is 2^-57
    ctx = dsbcg.Context(dims, torch.from_numpy(U).to(DEV), kappa)
    ctx.set_profiling(True)
    got = ctx.apply(op, torch.from_numpy(F[None]).to(DEV), storage="fp64").cpu().numpy()
    launches = ctx.read_profile()[1]
    ctx.close()
    assert launches["other"] == 1                             # converted: the fixed-point stencil ran
    terms = (np.abs(row) * np.sqrt(2)).sum() + 16.0
    assert abs(got[0, i] - want[0, i]) <= 32 * 2.0 ** -53 * terms
