"""The three-pass normal operator (spiral and 2-D masks) over its launch shapes.

The row passes run 512, 256 or 64 / 128 threads per block depending on the
number of row blocks in the launch (one image, a few, many); coil counts below
and above a step's coils, with a remainder.  One application agrees with the
FP64 oracle to 1e-5 (FP32 transforms: about 4 log2(L) roundings of 6e-8 per
value, and the FP32 point-spread sums), and an image's bits do not depend on
the batch it is in.
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

import synth
from oracle import ops as O

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("kind,n,nc", [("spiral", 32, 3), ("spiral", 40, 9), ("spiral", 64, 5), ("spiral", 120, 2),
                                       ("spiral", 160, 5), ("spiral", 240, 3), ("mask2d", 64, 17), ("mask2d", 96, 5),
                                       ("mask2d", 160, 9), ("mask2d", 192, 3), ("mask2d", 240, 1),
                                       ("mask2d", 320, 9), ("mask2d", 384, 5), ("mask2d", 480, 3)])
def test_normal_operator_launch_shapes(kind, n, nc):
    import paper_2605_09590_gb300 as pico
    rng = np.random.default_rng(n + nc)
    S = synth.coil_maps(n, n, nc, 3)
    kw = {}
    if kind == "spiral":
        kw["traj"] = synth.spiral_traj(n, 16, 64, 2)
    else:
        kw["mask"] = (rng.random((n, n)) < 0.5).astype(np.uint8)
    many = 304 * 4 // n + 2   # more row blocks than two per SM of a 152-SM part
    op = pico.Operator(S, max_batch=many, power_iters=0, **kw)
    x = (rng.standard_normal((many, n, n)) + 1j * rng.standard_normal((many, n, n))).astype(np.complex64)
    xd = torch.from_numpy(x).cuda()
    y = op.apply_normal(xd)
    few = max(1, many // 2)
    parts = [op.apply_normal(xd[:1].contiguous()), op.apply_normal(xd[:few].contiguous())]
    op.sync()
    assert torch.equal(y[:1], parts[0])
    assert torch.equal(y[:few], parts[1])
    for i in (0, many - 1):
        if kind == "spiral":
            want = O.ToeplitzNormal(S, kw["traj"]).apply(x[i].astype(np.complex128))
        else:
            want = O.cart_normal(x[i].astype(np.complex128), S.astype(np.complex128), kw["mask"])
        got = y[i].cpu().numpy()
        assert np.linalg.norm(got - want) <= 1e-5 * np.linalg.norm(want)
    op.close()
