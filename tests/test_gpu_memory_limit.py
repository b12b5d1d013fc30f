"""Calls that fit without the fixed-point buffers fit with them.

The links (576 bytes per site) and exponents of the fixed-point FP64 stencil
are an option, taken where the gauge field is in SU(3).  A context whose links
are off SU(3) by 1e-8 never takes them, so the least device memory with which
a call succeeds on it (found by bisection with dsbcg_debug_memory_limit, to
64 KB) must be enough on an SU(3) context too: the option goes before the call
fails.  Results are checked as usual: every true residual of a solve to tol, an
application to 64 x 2^-53 of the largest component against the unlimited call.
"""
import numpy as np
import pytest
import torch

from paper_1205_0359_gb300 import dsbcg, synth

pytestmark = pytest.mark.gpu
DEV = torch.device("cuda")
DIMS, M, S, TOL = (8, 8, 8, 8), 2, 2, 1e-10
SIGMA = np.array([0.1, 1.0])
STEP = 1 << 16


def _setup():
    rng = np.random.Generator(np.random.PCG64(17))
    U = synth.su3_links(DIMS, 0.4, rng)
    B = synth.gaussian_rhs(12 * synth.volume(DIMS), M, rng)
    return U, torch.from_numpy(B).to(DEV)


def _solve(ctx, B):
    X, st = ctx.solve(B, SIGMA, TOL, storage="fp64", raise_on_error=False)
    assert st["code"] in (0, -4), st["code"]
    if st["code"] == 0:
        assert st["true_relres"].max() <= TOL
    return st["code"]


def _apply(ctx, B, **kw):
    try:
        ctx.apply("A", B, storage="fp64", **kw)
        return 0
    except dsbcg.DSBCGError as e:
        assert e.code == -4
        return e.code


def _force(ctx, B):
    try:
        ctx.force(B[None], B[None], storage="fp64")
        return 0
    except dsbcg.DSBCGError as e:
        assert e.code == -4
        return e.code


CALLS = {"solve": _solve, "apply": _apply, "force": _force}


def _context(U, limit, prepare=None):
    ctx = dsbcg.Context(DIMS, torch.from_numpy(U).to(DEV), 0.12)
    if prepare is not None:
        prepare(ctx)
    ctx.debug_memory_limit(limit)
    return ctx


def _least(U, B, call):
    """Least limit (in steps) with which the call succeeds on a fresh context."""
    lo, hi = 0, 1 << 11                              # 128 MB
    while hi - lo > 1:
        mid = (lo + hi) // 2
        ctx = _context(U, mid * STEP)
        ok = call(ctx, B) == 0
        ctx.close()
        lo, hi = (lo, mid) if ok else (mid, hi)
    return hi * STEP


@pytest.mark.parametrize("name", ["solve", "apply", "force"])
@pytest.mark.parametrize("links_held", [False, True])
def test_su3_links_need_no_more_memory(name, links_held):
    U, B = _setup()
    call = CALLS[name]
    limit = _least(U * (1 + 1e-8), B, call)
    small = B[:1, :].contiguous()
    ctx = _context(U, limit, (lambda c: c.apply("D", small, storage="fp64")) if links_held else None)
    try:
        for _ in range(2):                           # a second call keeps to what the first one found
            assert call(ctx, B) == 0
        ctx.debug_memory_limit(-1)
        want = dsbcg.Context(DIMS, torch.from_numpy(U).to(DEV), 0.12)
        got, ref = ctx.apply("D", B, storage="fp64"), want.apply("D", B, storage="fp64")
        want.close()
        assert (got - ref).abs().max() <= 64 * 2.0 ** -53 * B.abs().max()
        # another shape is sized anew
        assert _solve(ctx, torch.cat([B, B.roll(1, 1)])) == 0
    finally:
        ctx.close()


def test_in_place_application_at_the_limit():
    """The held-back result of an overlapping call is an option too."""
    U, B = _setup()
    limit = _least(U * (1 + 1e-8), B, _apply)
    ctx = _context(U, -1)
    want = ctx.apply("A", B, storage="fp64")
    ctx.close()
    ctx = _context(U, limit)
    F = B.clone()
    assert _apply(ctx, F, out=F) == 0
    ctx.close()
    assert (F - want).abs().max() <= 4 * 64 * 2.0 ** -53 * B.abs().max()


def test_gauge_update_off_su3_gives_the_su3_copies_back():
    """FP64 and FP32 applications on SU(3) links hold fixed-point links (576 bytes
    per site) and 12-real ones (192); after an update to a field off SU(3) the
    device has that memory free again, to the 2 MB granularity of two blocks."""
    dims = (16, 16, 16, 16)
    V = synth.volume(dims)
    U = synth.su3_links(dims, 0.4, np.random.Generator(np.random.PCG64(5)))
    F = torch.ones((1, 12 * V), dtype=torch.complex128, device=DEV)
    off = torch.from_numpy(U * 1.01).to(DEV)
    ctx = dsbcg.Context(dims, torch.from_numpy(U).to(DEV), 0.12)
    try:
        for storage in ("fp64", "fp32"):
            ctx.apply("D", F, storage=storage)
        torch.cuda.synchronize()
        before = torch.cuda.mem_get_info()[0]
        ctx.update_gauge(off)
        assert torch.cuda.mem_get_info()[0] - before >= 768 * V - (4 << 20)
        ctx.update_gauge(torch.from_numpy(U).to(DEV))       # and back: both copies are made anew
        for storage in ("fp64", "fp32"):
            ctx.apply("D", F, storage=storage)
    finally:
        ctx.close()
