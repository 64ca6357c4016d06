"""The fused FISTA / tangent / adjoint iterations over image sides and level counts.

Sides whose bands are no multiple of a tile, bands of odd side (240 with four
levels: 15), one level, every level in the shared-memory core but the first, and
levels shorter than the filter (64 with five levels: side 4, the separate
passes).  Three iterations against the FP64 oracle: 1e-5 relative (FP32
transforms, three normal operators of about 1e-6 each).  Filters shorter than a
level only wrap once, so the oracle's periodic transform is the reference for
sides of at least 6.
"""
import numpy as np
import pytest

import synth
from oracle import cs as OCS
from oracle import ops as O

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def rel(a, b):
    return float(np.linalg.norm(a - b) / np.linalg.norm(b))


@pytest.mark.parametrize("n,levels", [(64, 1), (64, 4), (80, 3), (96, 4), (128, 2), (160, 4), (192, 5), (240, 4),
                                      (256, 3), (320, 1), (320, 2), (320, 4), (384, 6), (480, 3)])
def test_fused_iterations_match_oracle(n, levels):
    import paper_2605_09590_gb300 as pico
    rng = np.random.default_rng(n + levels)
    nc, nb, iters = 2, 3, 3
    S = synth.coil_maps(n, n, nc, 2)
    mask = (rng.random((n, n)) < 0.6).astype(np.uint8)
    oop = O.Operator(S, None, mask=mask)
    x0 = synth.phantom(n, 1).astype(np.complex128)
    b = oop.forward(x0)
    h, g = OCS.wavelet_filters(4)
    lam = 1e-2 * np.abs(OCS.dwt2(oop.adjoint(b), levels, h, g)).max()
    f = OCS.Fista(oop, b, lam, iters, levels=levels)
    op = pico.Operator(S, mask=mask, power_iters=15, max_batch=nb)
    dev = lambda a: torch.from_numpy(np.ascontiguousarray(a, dtype=np.complex64)).cuda()
    x = torch.empty((n, n), dtype=torch.complex64, device="cuda")
    pico.pico_cs_recon(op.ctx, dev(b), lam, iters, levels, x)
    db = ((rng.standard_normal((nb, nc, n, n)) + 1j * rng.standard_normal((nb, nc, n, n))) * mask).astype(np.complex64)
    xb = (rng.standard_normal((nb, n, n)) + 1j * rng.standard_normal((nb, n, n))).astype(np.complex64)
    dx = torch.empty((nb, n, n), dtype=torch.complex64, device="cuda")
    bb = torch.empty((nb, nc, n, n), dtype=torch.complex64, device="cuda")
    pico.pico_cs_jvp(op.ctx, dev(db), dx)
    pico.pico_cs_vjp(op.ctx, dev(xb), bb)
    one = torch.empty((1, n, n), dtype=torch.complex64, device="cuda")
    pico.pico_cs_jvp(op.ctx, dev(db[2:]), one)
    op.sync()
    assert rel(x.cpu().numpy(), f.x) < 1e-5
    assert torch.equal(one[0], dx[2])
    for i in (0, nb - 1):
        assert rel(dx[i].cpu().numpy(), f.jvp(db[i].astype(np.complex128))) < 1e-5
        assert rel(bb[i].cpu().numpy(), f.vjp(xb[i].astype(np.complex128))) < 1e-5
    op.close()


def test_levels_shorter_than_the_filter_still_run():
    import paper_2605_09590_gb300 as pico
    n = 64
    S = synth.coil_maps(n, n, 2, 2)
    op = pico.Operator(S, mask=np.ones((n, n), dtype=np.uint8), max_batch=2)
    b = op.forward(torch.ones((1, n, n), dtype=torch.complex64, device="cuda"))
    x = torch.empty((n, n), dtype=torch.complex64, device="cuda")
    pico.pico_cs_recon(op.ctx, b, 1e-3, 3, 5, x)
    op.sync()
    assert bool(torch.isfinite(torch.view_as_real(x)).all())
    op.close()
