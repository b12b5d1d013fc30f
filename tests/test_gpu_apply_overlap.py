"""dsbcg_apply with overlapping input and output.

The header does not promise it, but every storage reads all of `in` before it
writes `out`, so in-place and shifted calls give the result of separate
buffers.  That holds too when an FP64 call is repeated (fields that the fixed
point format does not hold: components far below the others, a NaN), for which
the input must still be there.
"""
import numpy as np
import pytest
import torch

from paper_1205_0359_gb300 import dsbcg, synth

pytestmark = pytest.mark.gpu
DIMS, M = (4, 4, 2, 4), 3


def _setup(kind):
    rng = np.random.Generator(np.random.PCG64(12))
    U = synth.su3_links(DIMS, 0.5, rng)
    F = synth.gaussian_rhs(12 * synth.volume(DIMS), M, rng).reshape(M, -1, 12)
    if kind == "graded":
        F[:, 5:] = 0
        F[:, 3, 4] *= 1e-15
    elif kind == "nan":
        F[1, 7, 2] = np.nan
    return dsbcg.Context(DIMS, torch.from_numpy(U).cuda(), 0.12), F.reshape(M, -1)


@pytest.mark.parametrize("where", ["device", "host", "pinned"])
@pytest.mark.parametrize("kind", ["dense", "graded", "nan"])
@pytest.mark.parametrize("op,storage", [("D", "fp64"), ("A", "fp64"), ("A", "fp32")])
@pytest.mark.parametrize("shift", [0, 1, -1])
def test_overlapping_buffers(where, kind, op, storage, shift):
    ctx, F = _setup(kind)
    want = ctx.apply(op, torch.from_numpy(F).cuda(), storage=storage).cpu().numpy()
    buf = torch.zeros((M + 1, F.shape[1]), dtype=torch.complex128)
    if where == "device":
        buf = buf.cuda()
    elif where == "pinned":
        buf = buf.pin_memory()
    a, b = (1, 1 + shift) if shift <= 0 else (0, 1)
    src, dst = buf[a:a + M], buf[b:b + M]
    src.copy_(torch.from_numpy(F))
    ctx.apply(op, src, storage=storage, out=dst)
    assert np.array_equal(dst.cpu().numpy(), want, equal_nan=True)
    ctx.close()
