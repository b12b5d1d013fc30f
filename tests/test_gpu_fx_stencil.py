"""The fixed-point FP64 stencil (links in SU(3)) against the oracle.

An application of D in block fixed point is exact to a few units of 2^-57 of
the largest component of a site and its eight neighbours, before the result
is rounded to FP64; the oracle's FP64 chains (3 x 3 products, eight hops)
carry about 10 x 2^-53 of it.  Every component therefore agrees with the
oracle to 32 x 2^-53 of the largest component of the site and its
neighbours (D), and twice that for A = D^H D, whose operator norm per hop
pair is below 4.
"""
import numpy as np
import pytest
import torch

from oracle import evenodd as EO
from oracle import wilson as W
from paper_1205_0359_gb300 import dsbcg, synth

pytestmark = pytest.mark.gpu
DEV = torch.device("cuda")
REF = {"D": W.D_vec, "Ddag": W.Ddag_vec, "A": W.A_vec}


def _fields(dims, m, seed, grade):
    """Gaussian fields, every site scaled by 10^-(0..grade)."""
    rng = np.random.Generator(np.random.PCG64(seed))
    V = synth.volume(dims)
    F = synth.gaussian_rhs(12 * V, m, rng).reshape(m, V, 12)
    return (F * 10.0 ** (-grade * rng.random((m, V, 1)))).reshape(m, 12 * V), synth.su3_links(dims, 0.7, rng)


def _site_max(F, dims, rings):
    """Largest component within `rings` hops of every site: (m, V, 1)."""
    m, (Lx, Ly, Lz, Lt) = F.shape[0], dims
    a = np.abs(F).reshape(m, Lt, Lz, Ly, Lx, 12).max(-1)
    for _ in range(rings):
        a = np.max([a] + [np.roll(a, s, axis=ax) for ax in (1, 2, 3, 4) for s in (1, -1)], axis=0)
    return a.reshape(m, -1, 1)


@pytest.mark.parametrize("dims", [(2, 2, 2, 2), (3, 5, 7, 4), (4, 4, 4, 8), (2, 4, 6, 5)])
@pytest.mark.parametrize("m", [1, 3, 4, 9])
@pytest.mark.parametrize("grade", [0, 12])
def test_every_component_to_its_neighbourhood(dims, m, grade):
    F, U = _fields(dims, m, 31 + m, grade)
    ctx = dsbcg.Context(dims, torch.from_numpy(U).to(DEV), 0.13)
    for op, ref in REF.items():
        got = ctx.apply(op, torch.from_numpy(F).to(DEV), storage="fp64").cpu().numpy()
        want = ref(U, 0.13, dims, F)
        bound = (64 if op == "A" else 32) * 2.0 ** -53 * _site_max(F, dims, 2 if op == "A" else 1)
        assert (np.abs(got - want).reshape(m, -1, 12) <= bound).all(), op
    ctx.close()


@pytest.mark.parametrize("kappa", [0.0, -0.11, 0.5, 3.0, 1e-12])
def test_kappa_range(kappa):
    """Any kappa: in the format's range (mantissa and exponent offset) or beyond it (FP64 kernels)."""
    dims, m = (4, 2, 4, 6), 3
    F, U = _fields(dims, m, 5, 0)
    ctx = dsbcg.Context(dims, torch.from_numpy(U).to(DEV), kappa)
    for op, ref in REF.items():
        got = ctx.apply(op, torch.from_numpy(F).to(DEV), storage="fp64").cpu().numpy()
        want = ref(U, kappa, dims, F)
        scale = (1.0 + 8.0 * abs(kappa)) ** (2 if op == "A" else 1)
        assert np.abs(got - want).max() <= 64 * 2.0 ** -53 * scale * np.abs(F).max(), op
    ctx.close()


@pytest.mark.parametrize("dims,m", [((4, 4, 4, 4), 2), ((2, 6, 4, 8), 5), ((6, 2, 2, 4), 1)])
def test_half_lattice(dims, m):
    rng = np.random.Generator(np.random.PCG64(3))
    U = synth.su3_links(dims, 0.7, rng)
    F = synth.gaussian_rhs(6 * synth.volume(dims), m, rng)
    ctx = dsbcg.Context(dims, torch.from_numpy(U).to(DEV), 0.13)
    ctx.set_operator("schur")
    for op, ref in (("D", EO.Dhat_vec), ("Ddag", EO.Dhat_dag_vec), ("A", EO.Ahat_vec)):
        got = ctx.apply(op, torch.from_numpy(F).to(DEV), storage="fp64").cpu().numpy()
        want = ref(U, 0.13, dims, F)
        assert np.abs(got - want).max() <= 128 * 2.0 ** -53 * np.abs(F).max(), op
    ctx.close()


@pytest.mark.parametrize("scale", [1e-300, 1e-230, 1e-120, 1e120, 1e260])
def test_extreme_magnitudes(scale):
    """Outside the range of the fixed-point format the FP64 kernels answer."""
    dims, m = (4, 4, 2, 4), 2
    F, U = _fields(dims, m, 8, 0)
    ctx = dsbcg.Context(dims, torch.from_numpy(U).to(DEV), 0.13)
    got = ctx.apply("A", torch.from_numpy(F * scale).to(DEV), storage="fp64").cpu().numpy()
    want = W.A_vec(U, 0.13, dims, F)
    assert np.abs(got / scale - want).max() <= 64 * 2.0 ** -53 * np.abs(F).max() + 24 * 5e-324 / scale
    ctx.close()


@pytest.mark.parametrize("value", [np.nan, np.inf, -np.inf])
def test_nonfinite_input_is_answered_by_the_fp64_kernels(value):
    """One non-finite component: finite and non-finite results are those of
    the oracle, component by component."""
    dims, m = (4, 4, 4, 4), 2
    F, U = _fields(dims, m, 9, 0)
    F[1, 12 * 37 + 5] = value
    ctx = dsbcg.Context(dims, torch.from_numpy(U).to(DEV), 0.13)
    got = ctx.apply("D", torch.from_numpy(F).to(DEV), storage="fp64").cpu().numpy()
    with np.errstate(invalid="ignore"):
        want = W.D_vec(U, 0.13, dims, F)
    fin = np.isfinite(want)
    assert np.isfinite(got[0]).all() and not np.isfinite(got[1]).all()
    # the oracle's dense gamma products spread a NaN at least as far
    assert np.isfinite(got[fin]).all()
    assert np.abs(got[fin] - want[fin]).max() <= 64 * 2.0 ** -53 * np.abs(F[np.isfinite(F)]).max()
    ctx.close()


def test_zero_sites_stay_zero():
    """A point source: D reaches the source and its eight neighbours, nothing else."""
    dims = (4, 6, 4, 8)
    V = synth.volume(dims)
    rng = np.random.Generator(np.random.PCG64(4))
    U = synth.su3_links(dims, 0.7, rng)
    F = np.zeros((1, 12 * V), dtype=complex)
    F[0, 12 * 100 + 3] = 1.0
    ctx = dsbcg.Context(dims, torch.from_numpy(U).to(DEV), 0.13)
    got = ctx.apply("D", torch.from_numpy(F).to(DEV), storage="fp64").cpu().numpy()
    want = W.D_vec(U, 0.13, dims, F)
    assert (np.abs(got).reshape(V, 12).max(-1) > 0).sum() == 9
    assert (got[np.abs(want) == 0] == 0).all() and np.abs(got - want).max() <= 32 * 2.0 ** -53
    ctx.close()
