"""CG solves over the batch sizes at which a launch changes its shape.

The on-chip solver takes 8, 16 or 32 images per block depending on how many
blocks stay resident, the column-FFT operator four instead of three blocks per
SM once a launch does not fit three.  A system's bits do not depend on its batch,
and one of them agrees with the oracle's CG (12 FP32 iterations from well
conditioned systems: 1e-5).
"""
import numpy as np
import pytest

import synth
from oracle import ops as O
from oracle import solvers

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("ny,nx,batches,solver", [
    (32, 30, (1, 40, 41, 90, 200), "global"), (32, 64, (2, 16, 17, 32, 33), "columns"),
    (64, 20, (8, 56, 57, 130), "global"), (64, 64, (3, 16, 17, 40), "columns"),
    (96, 50, (1, 24, 25, 60), "global"), (96, 33, (32, 33), "columns"),
    (192, 120, (3, 30, 31, 40), "global"), (240, 64, (8, 57, 58), "global"), (256, 64, (1, 57, 58, 60), "global"),
    (384, 40, (1, 20), "global")])
def test_bits_do_not_depend_on_the_launch_shape(ny, nx, batches, solver):
    import paper_2605_09590_gb300 as pico
    rng = np.random.default_rng(ny * nx)
    S = synth.coil_maps(ny, nx, 6, 7)
    mask = synth.mask_pe(ny, 2, 8)
    B = max(batches)
    op = pico.Operator(S, mask=mask, lam=0.05, max_batch=B)
    op.set_solver(solver)
    rhs = (rng.standard_normal((B, ny, nx)) + 1j * rng.standard_normal((B, ny, nx))).astype(np.complex64)
    rd = torch.from_numpy(rhs).cuda()
    full = op.cg(rd, 12)
    for nb in batches:
        assert torch.equal(op.cg(rd[:nb].contiguous(), 12), full[:nb])
    op.sync()
    if solver == "global":
        oop = O.Operator(S, None, mask=mask)
        lam = op.info["lambda_phys"]
        want, _, _ = solvers.cg_batched(lambda p: oop.normal(p[:, 0].reshape(ny, nx), lam).reshape(-1, 1),
                                        rhs[0].astype(np.complex128).reshape(-1, 1), 12)
        got = full[0].cpu().numpy().reshape(-1, 1)
        assert np.linalg.norm(got - want) <= 1e-5 * np.linalg.norm(want)
    op.close()
