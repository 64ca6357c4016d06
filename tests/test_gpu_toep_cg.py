"""CG on the three-pass operator (spiral and 2-D masks) over its launch shapes.

The row passes update the direction and sum p^H q in blocks of 512, 256 or
64 / 128 threads, by the number of row blocks in the launch.  Batches on each side
of both limits (one and two row blocks per SM): a system's bits do not depend on
its batch, and the first and last agree with the oracle's CG to the library's
parity bar of 1e-4 (12 iterations).
"""
import numpy as np
import pytest

import synth
from oracle import ops as O
from oracle import solvers

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("kind,n,nc", [("spiral", 32, 9), ("spiral", 64, 5), ("spiral", 120, 3), ("spiral", 160, 5),
                                       ("spiral", 240, 2), ("mask2d", 64, 9), ("mask2d", 96, 5), ("mask2d", 160, 3),
                                       ("mask2d", 240, 5), ("mask2d", 320, 3), ("mask2d", 480, 3)])
def test_bits_do_not_depend_on_the_batch(kind, n, nc):
    import paper_2605_09590_gb300 as pico
    rng = np.random.default_rng(n + nc)
    S = synth.coil_maps(n, n, nc, 3)
    kw = {}
    if kind == "spiral":
        kw["traj"] = synth.spiral_traj(n, 16, 64, 2)
        T = O.ToeplitzNormal(S, kw["traj"])
    else:
        kw["mask"] = (rng.random((n, n)) < 0.5).astype(np.uint8)
        T = None
    nsm = torch.cuda.get_device_properties(0).multi_processor_count
    per = n // 4                                     # row blocks of an image
    batches = sorted({max(1, nsm // per), nsm // per + 1, max(1, 2 * nsm // per), 2 * nsm // per + 1})
    op = pico.Operator(S, lam=0.1, power_iters=15, max_batch=batches[-1], **kw)
    lam = op.info["lambda_phys"]
    rhs = (rng.standard_normal((batches[-1], n, n)) + 1j * rng.standard_normal((batches[-1], n, n)))
    rhs = rhs.astype(np.complex64)
    rd = torch.from_numpy(rhs).cuda()
    full = op.cg(rd, 12)
    for nb in batches[:-1]:
        assert torch.equal(op.cg(rd[:nb].contiguous(), 12), full[:nb])
    op.sync()
    for i in (0, batches[-1] - 1):
        if T:
            apply = lambda z: T.apply(z, lam)  # noqa: E731
        else:
            apply = lambda z: O.cart_normal(z, S.astype(np.complex128), kw["mask"], lam)  # noqa: E731
        want, _, _ = solvers.cg(apply, rhs[i], 12)
        assert np.linalg.norm(full[i].cpu().numpy() - want) <= 1e-4 * np.linalg.norm(want)
    op.close()
