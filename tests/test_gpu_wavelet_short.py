"""Wavelet levels whose side is shorter than the 8-tap filter or close to it.

The transform is fully periodic: a side of 4 or 2 wraps more than once.  Sides of
6 are the shortest that the fused iterations take, 4 and 2 run the separate
passes.  The transform and its inverse against the FP64 oracle to 2e-6 (the bound
of the longer levels: 16 FMAs per value and level in FP32); reconstruction, JVP
and VJP of three iterations to 1e-5 as for the other sides; W^H W = 1 to 4e-6
(two transforms).
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


def dev(a):
    return torch.from_numpy(np.ascontiguousarray(a, dtype=np.complex64)).cuda()


def crandn(rng, *shape):
    return (rng.standard_normal(shape) + 1j * rng.standard_normal(shape)).astype(np.complex64)


@pytest.mark.parametrize("n,levels", [(32, 4), (32, 5), (48, 4), (64, 5), (64, 6), (96, 5), (128, 6), (128, 7),
                                      (192, 6), (384, 7)])
def test_transform_and_inverse_match_oracle(n, levels):
    import paper_2605_09590_gb300 as pico
    rng = np.random.default_rng(10 * n + levels)
    op = pico.Operator(synth.coil_maps(n, n, 1, 2), mask=synth.mask_pe(n, 2, 8), power_iters=0, max_batch=2)
    h, g = OCS.wavelet_filters(4)
    x = crandn(rng, 3, n, n)
    xd, c, back = dev(x), dev(x), dev(x)
    pico.pico_wavelet(op.ctx, xd, c, levels)
    pico.pico_wavelet(op.ctx, xd, back, levels, inverse=True)
    inv = back.cpu().numpy()
    pico.pico_wavelet(op.ctx, c, back, levels, inverse=True)
    op.sync()
    for i in range(3):
        assert rel(c[i].cpu().numpy(), OCS.dwt2(x[i].astype(np.complex128), levels, h, g)) < 2e-6
        assert rel(inv[i], OCS.idwt2(x[i].astype(np.complex128), levels, h, g)) < 2e-6
        assert rel(back[i].cpu().numpy(), x[i]) < 4e-6
    op.close()


@pytest.mark.parametrize("n,levels,mask2d", [(32, 4, False), (64, 5, True), (64, 6, True), (64, 6, False),
                                             (96, 5, True), (192, 6, True)])
def test_cs_iterations_match_oracle(n, levels, mask2d):
    import paper_2605_09590_gb300 as pico
    rng = np.random.default_rng(n + levels)
    nc, nb, iters = 2, 3, 3
    S = synth.coil_maps(n, n, nc, 2)
    mask = (rng.random((n, n)) < 0.6).astype(np.uint8) if mask2d else synth.mask_pe(n, 2, 8)
    sampled = mask if mask2d else np.asarray(mask)[:, None] * np.ones((1, n))
    oop = O.Operator(S, None, mask=mask)
    b = oop.forward(synth.phantom(n, 1).astype(np.complex128))
    h, g = OCS.wavelet_filters(4)
    lam = 1e-2 * np.abs(OCS.dwt2(oop.adjoint(b), levels, h, g)).max()
    f = OCS.Fista(oop, b, lam, iters, levels=levels)
    op = pico.Operator(S, mask=mask, power_iters=15, max_batch=nb)
    x = torch.empty((n, n), dtype=torch.complex64, device="cuda")
    pico.pico_cs_recon(op.ctx, dev(b), lam, iters, levels, x)
    db = (crandn(rng, nb, nc, n, n) * sampled).astype(np.complex64)
    xb = crandn(rng, nb, n, n)
    dx = torch.empty((nb, n, n), dtype=torch.complex64, device="cuda")
    bb = torch.empty((nb, nc, n, n), dtype=torch.complex64, device="cuda")
    pico.pico_cs_jvp(op.ctx, dev(db), dx)
    pico.pico_cs_vjp(op.ctx, dev(xb), bb)
    op.sync()
    assert rel(x.cpu().numpy(), f.x) < 1e-5
    for i in (0, nb - 1):
        assert rel(dx[i].cpu().numpy(), f.jvp(db[i].astype(np.complex128))) < 1e-5
        assert rel(bb[i].cpu().numpy(), f.vjp(xb[i].astype(np.complex128))) < 1e-5
    op.close()
