"""Launched-ahead block steps against plain launches, bitwise.

Small solves launch the kernels of a block step ahead of one another; with
the library's profiling on every launch is a plain one and the restarts run
one after another.  Each kernel does the same operations in the same order
either way, so solutions, residuals and step counts are bitwise the same: in
FP64 storage (conversion, fixed-point stencils, separate Gram, block update
and shift update; and, on links off SU(3), the FP64 stencil), in FP32 and
16-bit storage, with the even-odd operator, and through a deflation.
"""
import numpy as np
import pytest
import torch

from paper_1205_0359_gb300 import dsbcg, synth

pytestmark = pytest.mark.gpu
DEV = torch.device("cuda")


@pytest.mark.parametrize("storage,m,schur,su3", [
    ("fp64", 4, False, True), ("fp64", 11, False, True), ("fp64", 13, False, True), ("fp64", 4, False, False),
    ("fp64", 3, True, True), ("fp32", 5, False, True), ("fp32", 4, True, True), ("bf16", 4, False, True)])
def test_bitwise_equal_to_plain_launches(storage, m, schur, su3):
    dims = (4, 4, 6, 4) if schur else (3, 4, 5, 4)
    rng = np.random.Generator(np.random.PCG64(41 + m))
    U = synth.su3_links(dims, 0.4, rng)
    if not su3:
        U = U * (1.0 + 1e-6)
    B = synth.gaussian_rhs((6 if schur else 12) * synth.volume(dims), m, rng)
    B[m - 1] = B[0] + B[1]
    B = torch.from_numpy(B).to(DEV)
    sigma = synth.log_shifts(1e-2, 1.0, 3)
    ctx = dsbcg.Context(dims, torch.from_numpy(U).to(DEV), 0.12)
    try:
        if schur:
            ctx.set_operator("schur")
        Xa, sa = ctx.solve(B, sigma, 1e-10, storage=storage)
        ctx.set_profiling(True)
        Xp, sp = ctx.solve(B, sigma, 1e-10, storage=storage)
    finally:
        ctx.close()
    assert sa["code"] == sp["code"] == 0 and sa["deflations"] >= 1
    assert sa["block_steps"] == sp["block_steps"] and sa["restarts"] == sp["restarts"]
    assert torch.equal(Xa, Xp)
    assert np.array_equal(sa["true_relres"], sp["true_relres"])
