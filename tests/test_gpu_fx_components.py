"""FP64 applications, component by component.

Whatever the kernels compute in, an FP64 application is as good as an FP64
chain for EVERY complex component, small ones beside large ones included:

    |got - exact| <= C 2^-53 T,   T = |in| + |kappa| sum_hops |1 -+ gamma| |U| |in|

(all moduli, sums of non-negative terms; T of T for A = D^H D).  A chain of
FP64 operations is at most 16 roundings deep here and the oracle's about 24;
the fixed-point stencil may take 32 x 2^-53 of T, below which it leaves the
call to the FP64 kernels: C = 64, and 128 for the two passes of A.

Inputs: colours, spins and single components of a site graded over many
decades, on links that do not mix them (unit links, links of an SU(2)
subgroup, links with tiny off-diagonal entries), point sources, whole sites
graded, dense fields.
"""
import numpy as np
import pytest
import torch

from oracle import evenodd as EO
from oracle import wilson as W
from paper_1205_0359_gb300 import dsbcg, synth

pytestmark = pytest.mark.gpu
DEV = torch.device("cuda")
DIMS = (4, 2, 6, 4)
REF = {"D": W.D_vec, "Ddag": W.Ddag_vec, "A": W.A_vec}


def _links(kind, rng):
    V = synth.volume(DIMS)
    shape = DIMS[::-1] + (4,)
    unit = np.broadcast_to(np.eye(3, dtype=complex), shape + (3, 3)).copy()
    if kind == "unit":
        return unit
    if kind == "random":
        return synth.su3_links(DIMS, 0.7, rng)
    t = rng.uniform(0, 2 * np.pi, shape + (2,))
    if kind == "su2":                          # colours 0 and 1 mix, colour 2 does not
        c, s, p = np.cos(t[..., 0]), np.sin(t[..., 0]), np.exp(1j * t[..., 1])
        unit[..., 0, 0], unit[..., 0, 1] = c * p, s
        unit[..., 1, 0], unit[..., 1, 1] = -s, c * p.conj()
        return unit
    assert kind == "tiny"                      # phases, and off-diagonal entries of 1e-13
    ph = np.exp(1j * t)
    unit[..., 0, 0], unit[..., 1, 1], unit[..., 2, 2] = ph[..., 0], ph[..., 1], (ph[..., 0] * ph[..., 1]).conj()
    eps = 1e-13 * rng.standard_normal(shape + (3, 3))
    for a in range(3):
        eps[..., a, a] = 0
    return unit + eps


def _field(kind, m, rng):
    V = synth.volume(DIMS)
    F = synth.gaussian_rhs(12 * V, m, rng).reshape(m, V, 4, 3)
    if kind.startswith("colour"):              # the second colour far below the first, no third
        F[..., 1] *= 10.0 ** -int(kind[6:])
        F[..., 2] = 0
    elif kind == "one_colour":
        F[..., 1:] = 0
    elif kind == "spin":
        F[..., 1, :] *= 1e-10
        F[..., 2:, :] = 0
    elif kind == "site":                       # one site, every component of another size
        keep = F[:, 37].copy()
        F[:] = 0
        F[:, 37] = keep * 10.0 ** -(1.7 * np.arange(12).reshape(4, 3))
    elif kind == "point":
        F[:] = 0
        F[:, 21, 2, 1] = 1.0
    elif kind == "sites":
        F *= 10.0 ** (-12 * rng.random((m, V, 1, 1)))
    elif kind == "mixed":                      # small components beside large sites
        F *= 10.0 ** (-12 * rng.random((m, V, 4, 3)))
    else:
        assert kind == "dense"
    return F.reshape(m, 12 * V)


def _magnitudes(U, kappa, v, rounds):
    f = np.abs(W.to_field(v, DIMS))
    for _ in range(rounds):
        out = f.copy()
        for mu in range(4):
            P = np.abs(W.EYE4 - W.GAMMA[mu])
            for g, u in ((np.roll(f, -1, axis=-3 - mu), U[..., mu, :, :]), (np.roll(f, 1, axis=-3 - mu), W._link_backward(U, mu))):
                out += abs(kappa) * np.einsum("st,...ta->...sa", P, np.einsum("...ab,...sb->...sa", np.abs(u), g))
        f = out
    return W.to_vector(f)


@pytest.mark.parametrize("links", ["unit", "su2", "tiny", "random"])
@pytest.mark.parametrize("kind", ["dense", "colour8", "colour12", "colour18", "one_colour", "spin", "site", "point", "sites", "mixed"])
@pytest.mark.parametrize("kappa", [0.13, 0.0])
def test_every_component(links, kind, kappa):
    rng = np.random.Generator(np.random.PCG64(7))
    U, F = _links(links, rng), _field(kind, 5, rng)
    ctx = dsbcg.Context(DIMS, torch.from_numpy(U).to(DEV), kappa)
    for op, ref in REF.items():
        got = ctx.apply(op, torch.from_numpy(F).to(DEV), storage="fp64").cpu().numpy()
        n = 2 if op == "A" else 1
        err = np.abs(got - ref(U, kappa, DIMS, F)) / 2.0 ** -53
        T = _magnitudes(U, kappa, F, n)
        assert (err <= 64 * n * T).all(), (op, (err / np.maximum(T, 1e-300)).max())
    ctx.close()


@pytest.mark.parametrize("kind", ["dense", "colour8", "point"])
def test_half_lattice(kind):
    rng = np.random.Generator(np.random.PCG64(8))
    U = _links("su2", rng)
    odd = (np.indices(DIMS[::-1]).sum(0).reshape(-1) & 1) == 1
    F = _field(kind, 2, rng).reshape(2, -1, 12)[:, odd]
    full = np.zeros((2, odd.size, 12), dtype=complex)
    full[:, odd] = F
    ctx = dsbcg.Context(DIMS, torch.from_numpy(U).to(DEV), 0.13)
    ctx.set_operator("schur")
    got = ctx.apply("D", torch.from_numpy(F.reshape(2, -1)).to(DEV), storage="fp64").cpu().numpy().reshape(2, -1, 12)
    want = EO.Dhat_vec(U, 0.13, DIMS, F.reshape(2, -1)).reshape(2, -1, 12)
    # |in| + kappa^2 |H| |H| |in| on the odd sites, from two rounds on the whole lattice
    T = _magnitudes(U, 0.13, full.reshape(2, -1), 2).reshape(2, -1, 12)[:, odd]
    assert (np.abs(got - want) <= 128 * 2.0 ** -53 * T).all()
    ctx.close()
