"""Performance cases of the noise-map library: the calls that its users make.

Each case is a plain dict.  ``prepare`` builds what a user's program has in
hand (an ``Operator`` over one acquisition, k-space data or right-hand sides),
``run`` makes one pass through the public entry points, ``work`` counts the
bytes and floating-point operations of a pass that no implementation can do
without, and ``exact`` gives the same outputs in 64-bit arithmetic from plain
numpy / torch.

Acquisitions follow the library's own workloads: phase-encode Cartesian SENSE
(64 x 64 with 8 coils up to 320 x 320 with 15 correlated coils, the serving
mix's 192 ... 384 with 8 ... 32 coils), variable-density spirals (240 x 240,
20 coils, Tikhonov weight 0.1) and 2-D variable-density masks with the
L1-wavelet reconstruction (320 x 320, 15 coils).
"""
from __future__ import annotations

import math

import numpy as np
import torch

import paper_2605_09590_gb300 as pico

# image sizes the operators serve (phase-encode lines; spiral and 2-D-mask image sides)
PE_LINES = (32, 64, 96, 128, 160, 192, 240, 256, 320, 384)
SPIRAL_SIDES = (64, 80, 96, 120, 128, 160, 192, 240)
CS_SIDES = (128, 160, 192, 240, 256, 320, 384)
KINDS = {"phase": pico.PICO_PROBE_PHASE, "rademacher": pico.PICO_PROBE_RADEMACHER, "gauss": pico.PICO_PROBE_GAUSS}


def listed() -> list[dict]:
    return [
        # the smallest map: 64 x 64, 8 coils, 32 probes; interactive use, where latency counts
        dict(name="sense64_map", call="map", enc="pe", ny=64, nx=64, nc=8, R=2, acs=0, corr=False, lam=0.0,
             K=32, batch=32, iters=30, rtol=0.0, probe="phase", solver="global"),
        # a rectangular field of view, an odd coil count and a probe count that is no multiple of the batch
        dict(name="cart240x210_ragged_map", call="map", enc="pe", ny=240, nx=210, nc=11, R=2, acs=16, corr=True,
             lam=0.02, K=77, batch=64, iters=20, rtol=0.0, probe="rademacher", solver="global"),
        # the headline workload: 320 x 320, 15 correlated coils, R = 2 with 24 central lines, 256 probes
        dict(name="knee320_map", call="map", enc="pe", ny=320, nx=320, nc=15, R=2, acs=24, corr=True, lam=0.0,
             K=256, batch=256, iters=30, rtol=0.0, probe="phase", solver="global"),
        # its comparison arm: 256 pseudo replicas
        dict(name="knee320_pmr", call="pmr", enc="pe", ny=320, nx=320, nc=15, R=2, acs=24, corr=True, lam=0.0,
             K=256, batch=256, iters=30, rtol=0.0, sigma=1.0, solver="global"),
        # the same acquisition with CG per readout column
        dict(name="knee320_columns_map", call="map", enc="pe", ny=320, nx=320, nc=15, R=2, acs=24, corr=True,
             lam=0.0, K=128, batch=128, iters=30, rtol=0.0, probe="phase", solver="columns"),
        # image reconstruction of a small batch of right-hand sides to a tolerance (a slice group)
        dict(name="cart256_cg", call="cg", enc="pe", ny=256, nx=256, nc=8, R=2, acs=24, corr=False, lam=0.05,
             K=16, batch=16, iters=40, rtol=1e-4, typ_iters=12, solver="global"),
        # spiral map: 240 x 240, 20 coils, R = 2 of 16 interleaves, Tikhonov 0.1, 96 probes
        dict(name="spiral240_map", call="map", enc="spiral", ny=240, nx=240, nc=20, R=2, nsamp=4096, corr=False,
             lam=0.1, K=96, batch=96, iters=30, rtol=0.0, probe="phase", solver="global"),
        # spiral replicas at R = 4 under the usual stopping rule (at most 100 iterations, residual 1e-2)
        dict(name="spiral240_r4_pmr", call="pmr", enc="spiral", ny=240, nx=240, nc=20, R=4, nsamp=4096, corr=False,
             lam=0.1, K=32, batch=32, iters=100, rtol=1e-2, typ_iters=6, sigma=1e-2, solver="global"),
        # the encoding operator and its adjoint on a few images (simulation of k-space data)
        dict(name="spiral192_encode", call="encode", enc="spiral", ny=192, nx=192, nc=12, R=2, nsamp=2048,
             corr=True, lam=0.1, K=6, batch=8, solver="global"),
        # one L1-wavelet reconstruction, 100 FISTA iterations: a single image, launch-bound
        dict(name="cs320_recon", call="cs_recon", enc="mask2d", ny=320, nx=320, nc=15, R=2, acs=24, corr=True,
             lam=0.0, K=1, batch=8, fista=100, levels=4, lam_l1=0.2, solver="global"),
        # Jacobian noise map of that reconstruction, 48 probes
        dict(name="cs320_map", call="cs_map", enc="mask2d", ny=320, nx=320, nc=15, R=2, acs=24, corr=True,
             lam=0.0, K=48, batch=48, fista=100, levels=4, lam_l1=0.2, probe="phase", solver="global"),
        # replicas of a smaller nonlinear reconstruction, a count that is no multiple of the batch
        dict(name="cs256_pmr", call="cs_pmr", enc="mask2d", ny=256, nx=256, nc=12, R=2, acs=24, corr=True,
             lam=0.0, K=40, batch=32, fista=60, levels=3, lam_l1=0.2, sigma=2e-3, solver="global"),
    ]


def _log_int(rng, lo: int, hi: int) -> int:
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng) -> dict:
    """One more case of the same ranges."""
    call = rng.choice(("map", "map", "map", "pmr", "pmr", "cg", "encode", "cs_recon", "cs_map", "cs_pmr"))
    c = dict(call=call, corr=rng.random() < 0.5, solver="global")
    if call.startswith("cs"):
        c["enc"] = "mask2d"
    else:
        c["enc"] = rng.choice(("pe", "pe", "spiral"))
    c["nc"] = rng.randint(8, 32) if c["enc"] == "pe" else rng.randint(6, 20)
    if c["enc"] == "pe":
        c["ny"] = rng.choice(PE_LINES)
        if c["ny"] <= 96 or call in ("pmr", "encode"):
            c["nx"] = rng.choice([s for s in PE_LINES if s <= 2 * c["ny"]])
        else:
            c["nx"] = _log_int(rng, 48, 384)
        c.update(R=2, acs=rng.choice((0, 16, 24)), lam=rng.choice((0.02, 0.05, 0.1)))
        if call == "map" and c["ny"] >= 128:
            c["solver"] = rng.choice(("global", "columns"))
            if c["solver"] == "columns" and c["ny"] not in (128, 160, 192, 256, 320, 384):
                c["solver"] = "global"
    elif c["enc"] == "spiral":
        c["ny"] = c["nx"] = rng.choice(SPIRAL_SIDES)
        c.update(R=rng.choice((2, 3, 4)), nsamp=rng.choice((1024, 2048, 4096)), lam=rng.choice((0.05, 0.1)))
    else:
        c["levels"] = rng.choice((2, 3, 4))
        c["ny"] = c["nx"] = rng.choice(CS_SIDES)
        c.update(R=2, acs=24, lam=0.0, lam_l1=rng.choice((0.1, 0.2, 0.3)), fista=rng.choice((30, 60, 100)))
    c["K"] = {"cg": _log_int(rng, 1, 48), "encode": _log_int(rng, 1, 12), "cs_recon": 1,
              "cs_map": _log_int(rng, 4, 64), "cs_pmr": _log_int(rng, 4, 64)}.get(call) or _log_int(rng, 16, 256)
    if call in ("map", "pmr", "cg"):
        c.update(iters=rng.randint(8, 30), rtol=0.0)
    if call in ("map", "cs_map"):
        c["probe"] = rng.choice(("phase", "phase", "rademacher", "gauss"))
    if call in ("pmr", "cs_pmr"):
        c["sigma"] = 1e-2 if call == "pmr" else 2e-3
    limit = max(work(k)["flops"] for k in listed() if k["enc"] == c["enc"])
    while c["K"] > 1 and work(c)["flops"] > 0.9 * limit:
        c["K"] = c["K"] * 2 // 3
    c["batch"] = min(c["K"], rng.choice((32, 64, 128)))
    return c


# ---------------------------------------------------------------------------
# acquisitions (drawn from the seed alone)
# ---------------------------------------------------------------------------
def _coils(case: dict, rng) -> np.ndarray:
    """Smooth Gaussian-bump sensitivities on a circle around the image, sum |S|^2 = 1 per voxel."""
    ny, nx, nc = case["ny"], case["nx"], case["nc"]
    y = (np.arange(ny) - ny / 2)[:, None] / ny
    x = (np.arange(nx) - nx / 2)[None, :] / nx
    S = np.empty((nc, ny, nx), dtype=np.complex64)
    for c in range(nc):
        phi = 2 * math.pi * (c + rng.uniform(-0.25, 0.25)) / nc
        a, b, g = rng.uniform(-math.pi, math.pi, 3)
        cy, cx = 0.6 * math.sin(phi), 0.6 * math.cos(phi)
        ey = np.exp(-(y - cy) ** 2 / 0.245 + 2j * math.pi * b * y + 1j * g)
        ex = np.exp(-(x - cx) ** 2 / 0.245 + 2j * math.pi * a * x)
        S[c] = ey * ex
    S /= np.sqrt(np.sum(S.real ** 2 + S.imag ** 2, axis=0, keepdims=True))
    return S


def _noise_cov(nc: int, rng) -> np.ndarray:
    """Correlated channel noise: unit-modulus random-phase correlations of 0.5 / nc, unequal variances."""
    H = np.triu(np.exp(1j * rng.uniform(0, 2 * math.pi, (nc, nc))), 1)
    d = np.sqrt(rng.uniform(0.8, 1.2, nc))
    return d[:, None] * (np.eye(nc) + 0.5 / nc * (H + H.conj().T)) * d[None, :]


def _mask1d(case: dict) -> np.ndarray:
    ny, m = case["ny"], np.zeros(case["ny"], dtype=np.uint8)
    m[::case["R"]] = 1
    for k in range(-(case["acs"] // 2), case["acs"] // 2):
        m[k % ny] = 1
    return m


def _mask2d(case: dict, rng) -> np.ndarray:
    """Variable-density random mask with a fully sampled centre, about 1 / R of the grid (natural DFT order)."""
    n, h = case["ny"], case["acs"] // 2
    f = np.fft.fftfreq(n) * 2
    k = np.sqrt(f[:, None] ** 2 + f[None, :] ** 2) / math.sqrt(2)
    p = np.minimum(1.0, (1.6 - 1.4 * k) / case["R"])
    m = rng.random((n, n)) < p
    i = np.abs(np.fft.fftfreq(n) * n)
    m |= (i[:, None] <= h) & (i[None, :] <= h)
    return m.astype(np.uint8)


def _spiral(case: dict) -> np.ndarray:
    """Variable-density spiral, 16 interleaves of which every R-th is kept; cycles per field of view."""
    n, kmax, L = case["ny"], case["ny"] / 2, 16
    turns = math.ceil(1.5 * kmax / L)
    t = np.arange(case["nsamp"]) / (case["nsamp"] - 1)
    k = np.concatenate([kmax * t ** 1.5 * np.exp(2j * math.pi * (turns * t + l / L)) for l in range(0, L, case["R"])])
    k = np.stack([k.real, k.imag], axis=1)
    return np.where(k >= n / 2, k - n, k).astype(np.float32)


def _phantom(n: int, rng) -> np.ndarray:
    y = (np.arange(n) - n / 2)[:, None] / (n / 2)
    x = (np.arange(n) - n / 2)[None, :] / (n / 2)
    img = ((x / 0.75) ** 2 + (y / 0.9) ** 2 <= 1).astype(np.float64)
    for _ in range(9):
        cx, cy = rng.uniform(-0.5, 0.5, 2)
        ax, ay = rng.uniform(0.05, 0.3, 2)
        img[((x - cx) / ax) ** 2 + ((y - cy) / ay) ** 2 <= 1] += rng.uniform(-0.4, 0.4)
    return img * np.exp(0.3j * math.pi * (x + 0.5 * y))


def _inputs(case: dict, seed: int) -> dict:
    """Host-side acquisition and data of one seed."""
    rng = np.random.default_rng([seed, 0x9E37])
    a = {"smaps": _coils(case, rng), "noise_cov": _noise_cov(case["nc"], rng) if case["corr"] else None}
    if case["enc"] == "pe":
        a["mask"] = _mask1d(case)
    elif case["enc"] == "mask2d":
        a["mask"] = _mask2d(case, rng)
    else:
        a["traj"] = _spiral(case)
    shape = (case["K"], case["ny"], case["nx"])
    if case["call"] in ("cg", "encode"):
        z = rng.standard_normal(shape + (2,), dtype=np.float32)
        a["images"] = z[..., 0] + 1j * z[..., 1]
    if case["call"] == "encode":
        z = rng.standard_normal((case["K"], case["nc"], a["traj"].shape[0] if "traj" in a else shape[1] * shape[2], 2),
                                dtype=np.float32)
        y = z[..., 0] + 1j * z[..., 1]
        a["kspace"] = y if "traj" in a else y.reshape((case["K"], case["nc"]) + shape[1:])
    if case["call"].startswith("cs"):
        S = torch.from_numpy(_whiten(a)).to(_device())
        x = torch.from_numpy(_phantom(case["ny"], rng)).to(S)
        b = torch.fft.fft2(S * x, norm="ortho")
        z = rng.standard_normal(tuple(b.shape) + (2,), dtype=np.float32)
        b = b + 5e-3 * torch.from_numpy(z[..., 0] + 1j * z[..., 1]).to(b)  # receiver noise
        a["data"] = (b * torch.from_numpy(a["mask"]).to(b.device)).to(torch.complex64)
    return a


def _whiten(a: dict) -> np.ndarray:
    S = a["smaps"].astype(np.complex128)
    if a["noise_cov"] is None:
        return S
    Li = np.linalg.inv(np.linalg.cholesky(a["noise_cov"]))
    return np.tensordot(Li, S, axes=1)


def _device() -> str:
    return "cuda" if torch.cuda.is_available() else "cpu"


# ---------------------------------------------------------------------------
# the calls
# ---------------------------------------------------------------------------
def prepare(case: dict, seed: int) -> dict:
    a = _inputs(case, seed)
    op = pico.Operator(a["smaps"], mask=a.get("mask"), noise_cov=a["noise_cov"], traj=a.get("traj"),
                       lam=case["lam"], max_batch=case["batch"])
    if case["solver"] == "columns":
        op.set_solver("columns")
    st = {"case": case, "op": op, "seed": seed}
    for k in ("images", "kspace"):
        if k in a:
            st[k] = torch.from_numpy(a[k]).to("cuda")
    if "data" in a:
        st["data"] = a["data"]
        st["x"] = torch.empty((case["ny"], case["nx"]), dtype=torch.complex64, device="cuda")
        if case["call"] != "cs_recon":  # maps are taken at a reconstruction
            pico.pico_cs_recon(op.ctx, st["data"], case["lam_l1"], case["fista"], case["levels"], st["x"])
    return st


def run(st: dict):
    case, op, seed = st["case"], st["op"], st["seed"]
    call = case["call"]
    if call == "map":
        s, ss = op.variance_sums(seed, case["K"], case["iters"], case["rtol"], kind=KINDS[case["probe"]])
        return (s, ss) + op.finalize(s, ss, case["K"])
    if call == "pmr":
        s, ss = op.pmr_sums(seed, case["K"], case["sigma"], case["iters"], case["rtol"])
        return (s, ss) + op.finalize(s, ss, case["K"])
    if call == "cg":
        return op.cg(st["images"], case["iters"], case["rtol"])
    if call == "encode":
        return op.forward(st["images"]), op.adjoint(st["kspace"])
    if call == "cs_recon":
        pico.pico_cs_recon(op.ctx, st["data"], case["lam_l1"], case["fista"], case["levels"], st["x"])
        return st["x"]
    s = torch.empty((case["ny"], case["nx"]), dtype=torch.float64, device="cuda")
    ss = torch.empty_like(s)
    if call == "cs_map":
        pico.pico_cs_variance_map(op.ctx, seed, 0, case["K"], KINDS[case["probe"]], s, ss)
    else:
        pico.pico_cs_pmr(op.ctx, seed, 0, case["K"], case["sigma"], s, ss)
    return (s, ss) + op.finalize(s, ss, case["K"])


def work(case: dict) -> dict:
    ny, nx, nc, K, enc, call = (case[k] for k in ("ny", "nx", "nc", "K", "enc", "call"))
    n = ny * nx
    fft = lambda N: 5.0 * N * math.log2(N)
    samples = math.ceil(16 / case["R"]) * case["nsamp"] if enc == "spiral" else n
    kspace = nc * samples
    if enc == "pe":       # column transforms: the mask leaves the readout direction alone
        normal = nc * nx * (2 * fft(ny) + 16 * ny)
        adjoint = nc * (ny / case["R"] * fft(nx) + nx * fft(ny) + 8 * n)
    elif enc == "mask2d":
        normal = nc * (2 * (ny * fft(nx) + nx * fft(ny)) + 18 * n)
        adjoint = nc * (ny * fft(nx) + nx * fft(ny) + 8 * n)
    else:                 # Toeplitz embedding on the doubled grid; Kaiser-Bessel gridding of width 6
        L = 2 * ny
        normal = nc * ((2 * ny + 2 * L) * fft(L) + 16 * n + 2 * L * L)
        adjoint = nc * ((L + ny) * fft(L) + 8 * n + 4 * 36 * samples)
    vec = 34.0 * n        # CG vector arithmetic of one iteration
    io = nc * n * 8.0
    if call in ("map", "pmr", "cg"):
        it = case.get("typ_iters", case["iters"])
        solve = it * (normal + vec)
        if call == "map":
            flops = K * (solve if case["lam"] == 0 else 2 * solve + normal)
        else:
            flops = K * (solve + (adjoint if call == "pmr" else 0.0))
        io += 2 * 8.0 * n * K if call == "cg" else 24.0 * n
    elif call == "encode":
        flops = 2.0 * K * adjoint
        io += 2 * 8.0 * K * (n + kspace)
    else:
        dwt = 4.0 / 3 * 2 * 2 * 8 * 2 * n   # one 2-D transform, all levels: 8 real taps both ways
        it = case["fista"] * (normal + 2 * dwt + 24.0 * n)
        flops = {"cs_recon": it + adjoint, "cs_map": K * (2 * it + normal), "cs_pmr": K * (it + adjoint)}[call]
        io += 8.0 * (kspace + n) if call == "cs_recon" else 24.0 * n
    return {"bytes": io, "flops": flops}


# ---------------------------------------------------------------------------
# the same outputs in 64 bits
# ---------------------------------------------------------------------------
def _i64(v: int) -> int:
    return v - (1 << 64) if v >= 1 << 63 else v


_G, _A, _B = _i64(0x9E3779B97F4A7C15), _i64(0xBF58476D1CE4E5B9), _i64(0x94D049BB133111EB)


def _shr(z, k: int):
    return (z >> k) & ((1 << (64 - k)) - 1)


def _splitmix(state, i):
    """Output i of SplitMix64 seeded with state (int64 tensors, wrapping arithmetic)."""
    z = state + (i + 1) * _G
    z = (z ^ _shr(z, 30)) * _A
    z = (z ^ _shr(z, 27)) * _B
    return z ^ _shr(z, 31)


def _key(seed: int, p: int, dev):
    return _splitmix(torch.tensor(seed, dtype=torch.int64, device=dev), torch.tensor(p, dtype=torch.int64, device=dev))


def _polar(r, h):
    return torch.polar(r, 2 * math.pi * 2.0 ** -24 * _shr(h, 40).to(torch.float64))


def _gauss(key, e):
    u = (_shr(_splitmix(key, 2 * e), 40).to(torch.float64) + 1) * 2.0 ** -24
    return _polar(torch.sqrt(-torch.log(u)), _splitmix(key, 2 * e + 1))


def _probe(seed: int, p: int, n: int, kind: str, dev):
    key, e = _key(seed, p, dev), torch.arange(n, dtype=torch.int64, device=dev)
    if kind == "gauss":
        return _gauss(key, e)
    h = _splitmix(key, 2 * e)
    if kind == "rademacher":
        return (1.0 - 2.0 * _shr(h, 63).to(torch.float64)).to(torch.complex128)
    return _polar(torch.ones(n, dtype=torch.float64, device=dev), h)


class _Exact:
    """The encoding operator of one case in complex128."""

    def __init__(self, case, seed):
        self.case, self.a, self.dev = case, _inputs(case, seed), _device()
        self.S = torch.from_numpy(_whiten(self.a)).to(self.dev)
        self.nc, self.ny, self.nx = self.S.shape
        self.enc, L = case["enc"], 2 * self.ny
        if self.enc == "spiral":
            k = torch.from_numpy(self.a["traj"].astype(np.float64)).to(self.dev)
            n, d = self.ny, torch.arange(self.ny, dtype=torch.float64, device=self.dev)
            lag = torch.arange(-(n - 1), n, dtype=torch.float64, device=self.dev)
            wave = lambda kk, r: torch.polar(torch.ones((), dtype=torch.float64, device=self.dev),
                                             -2 * math.pi / n * kk[:, None] * r[None, :])
            self.ey, self.ex = wave(k[:, 1], d) / math.sqrt(n), wave(k[:, 0], d) / math.sqrt(n)
            h = wave(k[:, 1], lag).conj().T @ wave(k[:, 0], lag).conj() / n ** 2
            C = torch.zeros((L, L), dtype=torch.complex128, device=self.dev)
            i = (torch.arange(-(n - 1), n, device=self.dev)) % L
            C[i[:, None], i[None, :]] = h
            self.T = torch.fft.fft2(C)
        else:
            m = torch.from_numpy(self.a["mask"]).to(self.dev).to(torch.float64)
            self.m = m[:, None].expand(self.ny, self.nx) if m.ndim == 1 else m
        self.lmax = None

    def normal(self, x, lam=0.0):
        out = lam * x
        for c in range(self.nc):
            z = self.S[c] * x
            if self.enc == "pe":
                z = torch.fft.ifft(torch.fft.fft(z, dim=-2) * self.m, dim=-2)
            elif self.enc == "mask2d":
                z = torch.fft.ifft2(torch.fft.fft2(z) * self.m)
            else:
                L = 2 * self.ny
                z = torch.fft.ifft2(torch.fft.fft2(z, s=(L, L)) * self.T)[..., :self.ny, :self.nx]
            out = out + self.S[c].conj() * z
        return out

    def forward(self, x):
        z = self.S[None] * x[:, None]
        if self.enc == "spiral":
            return torch.stack([torch.stack([((zc @ self.ex.T) * self.ey.T).sum(0) for zc in zb]) for zb in z])
        return torch.fft.fft2(z, norm="ortho") * self.m

    def adjoint(self, y):
        if self.enc == "spiral":
            return torch.stack([sum(self.S[c].conj() * ((self.ey.conj().T * yb[c][None]) @ self.ex.conj())
                                    for c in range(self.nc)) for yb in y])
        return (self.S.conj()[None] * torch.fft.ifft2(y * self.m, norm="ortho")).sum(1)

    def lambda_max(self):
        if self.lmax is None:
            n = self.ny * self.nx
            x = _probe(0x50574D, 0, n, "phase", self.dev).reshape(1, self.ny, self.nx) / math.sqrt(n)
            for _ in range(15):
                y = self.normal(x)
                self.lmax = float(torch.linalg.vector_norm(y))
                x = y / self.lmax
        return self.lmax

    def cg(self, b, iters, rtol, lam, columns):
        dims = (-2,) if columns else (-2, -1)
        dot = lambda u, v: (u.real * v.real + u.imag * v.imag).sum(dims, keepdim=True)
        x, r, p = torch.zeros_like(b), b.clone(), b.clone()
        rr = dot(r, r)
        stop = rtol ** 2 * rr
        for _ in range(iters):
            live = rr > stop
            if not bool(live.any()):
                break
            q = self.normal(p, lam)
            al = torch.where(live, rr / dot(p, q), torch.zeros_like(rr))
            x, r = x + al * p, r - al * q
            new = torch.where(live, dot(r, r), rr)
            p = torch.where(live, r + (new / rr) * p, p)
            rr = new
        return x

    def probes(self, seed, lo, hi, kind):
        v = torch.stack([_probe(seed, p, self.ny * self.nx, kind, self.dev) for p in range(lo, hi)])
        return v.reshape(hi - lo, self.ny, self.nx)

    def noise(self, seed, lo, hi, sigma):
        per = self.a["traj"].shape[0] if self.enc == "spiral" else self.ny * self.nx
        e = torch.arange(self.nc * per, dtype=torch.int64, device=self.dev)
        z = torch.stack([sigma * _gauss(_key(seed, p, self.dev), e) for p in range(lo, hi)])
        shape = (per,) if self.enc == "spiral" else (self.ny, self.nx)
        return z.reshape((hi - lo, self.nc) + shape)


# db4 scaling filter (Daubechies 1988, Table 1) and its quadrature mirror
_H = (0.2303778133088964, 0.7148465705529154, 0.6308807679298587, -0.0279837694168599,
      -0.1870348117190931, 0.0308413818355607, 0.0328830116668852, -0.0105974017850690)


def _dwt1(n, dev):
    W = np.zeros((n, n))
    for k in range(n // 2):
        for m in range(8):
            W[k, (2 * k + m) % n] += _H[m]
            W[n // 2 + k, (2 * k + m) % n] += (-1) ** m * _H[7 - m]
    return torch.from_numpy(W).to(dev).to(torch.complex128)


class _Fista:
    """L1-wavelet FISTA with its tangent and adjoint in complex128."""

    def __init__(self, E: _Exact):
        self.E, c = E, E.case
        self.lc = 1.01 * E.lambda_max()
        self.tau, self.iters = c["lam_l1"] / self.lc, c["fista"]
        self.W = [_dwt1(c["ny"] >> l, E.dev) for l in range(c["levels"])]
        self.cs, t = [], 1.0
        for _ in range(self.iters):
            tn = 0.5 * (1 + math.sqrt(1 + 4 * t * t))
            self.cs.append((t - 1) / tn)
            t = tn

    def dwt(self, x):
        x = x.clone()
        for W in self.W:
            m = W.shape[0]
            x[..., :m, :m] = W @ x[..., :m, :m] @ W.T
        return x

    def idwt(self, x):
        x = x.clone()
        for W in reversed(self.W):
            m = W.shape[0]
            x[..., :m, :m] = W.T @ x[..., :m, :m] @ W
        return x

    def recon(self, ahb, keep=False):
        x = z = torch.zeros_like(ahb)
        self.at = []
        for k in range(self.iters):
            w = self.dwt(z - (self.E.normal(z) - ahb) / self.lc)
            if keep:
                self.at.append(w)
            w = w * (1 - self.tau / w.abs().clamp_min(self.tau))
            xn = self.idwt(w)
            x, z = xn, xn + self.cs[k] * (xn - x)
        return x

    def _tan(self, k, d):
        a = self.at[k].abs()
        on, a = a > self.tau, a.clamp_min(self.tau)
        u = self.at[k] / a
        re = u.real * d.real + u.imag * d.imag
        return torch.where(on, (1 - self.tau / a) * d + (self.tau / a) * re * u, torch.zeros_like(d))

    def jjt(self, v):
        ys, zb, xb = torch.zeros_like(v), torch.zeros_like(v), v
        for k in reversed(range(self.iters)):
            xk, xb = xb + (1 + self.cs[k]) * zb, -self.cs[k] * zb
            yb = self.idwt(self._tan(k, self.dwt(xk)))
            zb, ys = yb - self.E.normal(yb) / self.lc, ys + yb
        g = self.E.normal(ys / self.lc)
        dx = dz = torch.zeros_like(v)
        for k in range(self.iters):
            w = self._tan(k, self.dwt(dz - (self.E.normal(dz) - g) / self.lc))
            xn = self.idwt(w)
            dx, dz = xn, xn + self.cs[k] * (xn - dx)
        return dx


def _finish(s, ss, K):
    m = s / K
    se = torch.sqrt(torch.clamp(ss / K - m * m, min=0) / (K - 1)) if K > 1 else torch.zeros_like(m)
    return s, ss, m, se


def exact(case: dict, seed: int):
    call, K = case["call"], case["K"]
    if case["enc"] == "spiral" and call in ("pmr", "encode"):
        samples = 16 / case["R"] * case["nsamp"] * case["nc"] * K
        if samples * 8 * case["ny"] ** 2 > 8e12:  # exact transforms of every sample: too long
            return None
    E = _Exact(case, seed)
    if call == "encode":
        return (E.forward(torch.from_numpy(E.a["images"]).to(E.S)), E.adjoint(torch.from_numpy(E.a["kspace"]).to(E.S)))
    lam = case["lam"] * 1.01 * E.lambda_max() if case["lam"] else 0.0
    columns = case["solver"] == "columns"
    if call == "cg":
        return E.cg(torch.from_numpy(E.a["images"]).to(E.S), case["iters"], case["rtol"], lam, columns)
    if call.startswith("cs"):
        F = _Fista(E)
        ahb = E.adjoint(E.a["data"].to(torch.complex128)[None])
        x0 = F.recon(ahb, keep=call == "cs_map")
        if call == "cs_recon":
            return x0[0]
    s = torch.zeros((E.ny, E.nx), dtype=torch.float64, device=E.dev)
    ss = torch.zeros_like(s)
    for lo in range(0, K, 32):
        hi = min(K, lo + 32)
        if call in ("map", "cs_map"):
            v = E.probes(seed, lo, hi, case["probe"])
            if call == "map":
                u = E.cg(v, case["iters"], case["rtol"], lam, columns)
                if lam:
                    u = E.cg(E.normal(u), case["iters"], case["rtol"], lam, columns)
            else:
                u = F.jjt(v)
            d = v.real * u.real + v.imag * u.imag
        else:
            rhs = torch.cat([E.adjoint(E.noise(seed, i, i + 1, case["sigma"])) for i in range(lo, hi)])
            if call == "pmr":
                u = E.cg(rhs, case["iters"], case["rtol"], lam, columns)
            else:
                u = F.recon(ahb + rhs) - x0
            d = (u.real ** 2 + u.imag ** 2) / case["sigma"] ** 2
        s, ss = s + d.sum(0), ss + (d * d).sum(0)
    return _finish(s, ss, K)
