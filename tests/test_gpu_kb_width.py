"""Gridding and interpolation at every window width the library takes (2, 4, 6, 8).

Against a dense FP64 model of the same Kaiser-Bessel transform (window,
deapodisation, oversampling 2), so that the narrow windows' aliasing is on both
sides.  FP32 bounds: a weight is a Bessel function of beta sqrt(1 - t^2) with
beta <= 18.6, whose argument carries about 1.2e-7 relative, 2.5e-6 per dimension;
with the transforms (4 log2(L) roundings of 6e-8) 1e-5 relative is allowed.
At width 8 the model itself agrees with the exact NUDFT to 1e-5.
Samples: uniform over the band, on grid points and half-way between them (windows
that end on a grid point), and at the band's corner, where windows wrap.
"""
import numpy as np
import pytest

import synth
from oracle import ops as O

torch = pytest.importorskip("torch")


class KaiserBessel:
    def __init__(self, traj, n, width):
        self.n, self.L = n, 2 * n
        beta = np.pi * np.sqrt((width / 2) ** 2 * 1.5 ** 2 - 0.8)
        nu = (np.arange(n) - n // 2) / self.L
        z = np.sqrt(beta ** 2 - (np.pi * width * nu) ** 2)   # positive: width |nu| <= 2 < beta / pi
        self.d = np.i0(beta) * z / (width * np.sinh(z)) / np.sqrt(n)
        self.w = []
        for u in (2 * traj).T:   # x, y; FP32 positions are exact
            w = np.zeros((len(u), self.L))
            for k in range(-1, width + 2):
                g = np.floor(u - np.float32(width / 2)) + k
                t = (g.astype(np.float32) - u).astype(np.float64) / (width / 2)
                v = np.where(np.abs(t) <= 1, np.i0(beta * np.sqrt(np.maximum(0, 1 - t * t))) / np.i0(beta), 0)
                np.add.at(w, (np.arange(len(u)), g.astype(int) % self.L), v)
            self.w.append(w)
        self.phase = np.exp(1j * np.pi * traj.astype(np.float64).sum(1))
        self.at = (np.arange(n) - n // 2) % self.L

    def forward(self, z):
        grid = np.zeros((self.L, self.L), dtype=complex)
        grid[np.ix_(self.at, self.at)] = z * np.outer(self.d, self.d)
        f = np.fft.fft2(grid)
        return np.conj(self.phase) * np.einsum("my,yx,mx->m", self.w[1], f, self.w[0], optimize=True)

    def adjoint(self, y):
        grid = (self.w[1] * (y * self.phase)[:, None]).T @ self.w[0]
        f = np.fft.ifft2(grid) * self.L ** 2
        return f[np.ix_(self.at, self.at)] * np.outer(self.d, self.d)


def trajectory(n, rng):
    h = n // 2
    grid = rng.integers(-2 * h, 2 * h, (60, 2)) / 2.0
    half = (rng.integers(-2 * h, 2 * h - 1, (60, 2)) + 0.5) / 2.0
    edge = np.array([[-h, -h], [h - 0.25, -h], [-h, h - 0.25], [h - 0.25, h - 0.25], [0, 0], [-0.125, 0.125]])
    return np.concatenate([rng.uniform(-h, h, (400, 2)), grid, half, edge]).astype(np.float32)


def crandn(rng, *shape):
    return (rng.standard_normal(shape) + 1j * rng.standard_normal(shape)).astype(np.complex64)


def rel(a, b):
    return np.linalg.norm(a - b) / np.linalg.norm(b)


def test_model_agrees_with_the_exact_nudft():
    rng = np.random.default_rng(1)
    n = 32
    traj = trajectory(n, rng)
    kb, exact = KaiserBessel(traj, n, 8), O.Nudft(traj, n)
    z, y = crandn(rng, n, n).astype(complex), crandn(rng, len(traj)).astype(complex)
    assert rel(kb.forward(z), exact.forward(z)) < 1e-5
    assert rel(kb.adjoint(y), exact.adjoint(y)) < 1e-5


@pytest.mark.gpu
@pytest.mark.parametrize("n,nc", [(32, 5), (40, 13), (64, 9), (96, 4)])
@pytest.mark.parametrize("width", [2, 4, 6, 8])
def test_every_window_width(n, nc, width):
    import paper_2605_09590_gb300 as pico
    rng = np.random.default_rng(100 * n + width)
    S = synth.coil_maps(n, n, nc, 4)
    traj = trajectory(n, rng)
    kb = KaiserBessel(traj, n, width)
    op = pico.Operator(S, traj=traj, power_iters=0, max_batch=2, kb_width=width)
    x, y = crandn(rng, 2, n, n), crandn(rng, 2, nc, len(traj))
    k = op.forward(torch.from_numpy(x).cuda()).cpu().numpy()
    a = op.adjoint(torch.from_numpy(y).cuda()).cpu().numpy()
    op.sync()
    op.close()
    for i in range(2):
        assert rel(k[i], np.stack([kb.forward(S[c] * x[i].astype(complex)) for c in range(nc)])) < 1e-5
        assert rel(a[i], sum(np.conj(S[c]) * kb.adjoint(y[i, c].astype(complex)) for c in range(nc))) < 1e-5
