"""Spiral gridding and interpolation over coil counts and grid splits.

The gridding kernel takes 4, 8, 10 or 12 coils per block and the interpolation
four per thread, with a remainder; every grid split has its own row and column
passes.  Against the exact NUDFT of the FP64 oracle: the Kaiser-Bessel window
(W = 6, oversampling 2) is accurate to about 1e-5; 2e-5 is allowed.
"""
import numpy as np
import pytest

import synth
from oracle import ops as O

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,nc", [(32, 1), (40, 5), (48, 8), (64, 9), (64, 13), (80, 10), (96, 12), (120, 3),
                                  (128, 11), (160, 2), (192, 20), (240, 4)])
def test_forward_and_adjoint_match_exact_nudft(n, nc):
    import paper_2605_09590_gb300 as pico
    rng = np.random.default_rng(n + nc)
    S = synth.coil_maps(n, n, nc, 4)
    traj = synth.spiral_traj(n, 4, 150, 1)
    op = pico.Operator(S, traj=traj, power_iters=0, max_batch=2)
    oop = O.Operator(S, None, traj=traj)
    x = (rng.standard_normal((2, n, n)) + 1j * rng.standard_normal((2, n, n))).astype(np.complex64)
    y = (rng.standard_normal((2, nc, len(traj))) + 1j * rng.standard_normal((2, nc, len(traj)))).astype(np.complex64)
    k = op.forward(torch.from_numpy(x).cuda()).cpu().numpy()
    a = op.adjoint(torch.from_numpy(y).cuda()).cpu().numpy()
    op.sync()
    op.close()
    for i in range(2):
        want = oop.forward(x[i].astype(np.complex128))
        assert np.linalg.norm(k[i] - want) < 2e-5 * np.linalg.norm(want)
        want = oop.adjoint(y[i].astype(np.complex128))
        assert np.linalg.norm(a[i] - want) < 2e-5 * np.linalg.norm(want)
