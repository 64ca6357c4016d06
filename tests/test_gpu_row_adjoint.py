"""Cartesian row adjoint over image widths and batches.

Few row blocks take 16-row blocks, many take four-row blocks of several coils
per step; coil counts leave a remainder.  One adjoint agrees with the FP64 oracle
to 2e-6 (the bound of the other Cartesian encoding tests), and an image's bits do
not depend on the batch it is in.
"""
import numpy as np
import pytest

import synth
from oracle import ops as O

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("ny,nx,nc", [(32, 64, 3), (40, 48, 5), (64, 80, 9), (96, 120, 4), (120, 96, 7), (128, 128, 3),
                                      (160, 160, 5), (192, 192, 1), (256, 240, 3), (240, 256, 2), (320, 320, 5),
                                      (32, 384, 3)])
def test_row_adjoint_batches(ny, nx, nc):
    import paper_2605_09590_gb300 as pico
    rng = np.random.default_rng(ny + nx + nc)
    S = synth.coil_maps(ny, nx, nc, 6)
    mask = synth.mask_pe(ny, 2, 8)
    many = 304 * 4 // ny + 2   # more four-row blocks than two per SM of a 152-SM part
    op = pico.Operator(S, mask=mask, power_iters=0, max_batch=many)
    oop = O.Operator(S, None, mask=mask)
    y = (rng.standard_normal((many, nc, ny, nx)) + 1j * rng.standard_normal((many, nc, ny, nx))).astype(np.complex64)
    yd = torch.from_numpy(y).cuda()
    x = op.adjoint(yd)
    one = op.adjoint(yd[-1:].contiguous())
    op.sync()
    assert torch.equal(one[0], x[-1])
    for i in (0, many - 1):
        want = oop.adjoint(y[i].astype(np.complex128))
        got = x[i].cpu().numpy()
        assert np.linalg.norm(got - want) < 2e-6 * np.linalg.norm(want)
    op.close()
