"""The work a user of the map-making library has it do, as cases that can be timed.

Every case goes through ``paper_1801_08937_gb300.mapmaker.Context``: operator
products, right-hand sides, template-filtered products, preconditioner calls,
a new scan's set-up, a coarse space, and whole solves.  The scans are the
back-and-forth rasters of the benchmark's workloads (0.14 pixel per sample,
half-wave-plate angle uniform in [0, pi), 1/f noise stationary per block),
made on the device from a seed.

``exact`` gives the same results in 64 bits with plain torch: the pointing by
indexing, the banded Toeplitz weight by zero-padded FFTs, the templates by
orthogonal projections, and solves by PCG run to rounding level.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_1801_08937_gb300 import mapmaker as M

DEV = "cuda"
FS_HZ = 100.0          # sampling rate
SPEED_PX = 0.14        # raster speed, pixels per sample
AZ_BIN_PX = 2.82       # azimuth bin of the ground template, pixels
RCOND_MIN = 1e-3


def listed():
    return [
        # One product with A on the small float64 problem (32x32 patch, 8 detectors x 32768 samples,
        # lambda 512): what each step of an interactive solve or an Arnoldi process calls.
        dict(name="A_small_fp64", kind="apply", prec="fp64", nx=32, n_det=8, n_t=32768, block=4096, half_bw=512,
             n_bands=8, nrhs=1, ragged=False, flagged=0.0),
        # The same problem solved to 1e-8 with M_BD from a device timeline: the smallest whole map.
        dict(name="solve_small_fp64", kind="solve", prec="fp64", nx=32, n_det=8, n_t=32768, block=4096, half_bw=512,
             n_bands=8, nrhs=1, uneven=False, two_level=False, tol=1e-8, max_iter=500, products=40, graphs=False),
        # Coarse-space set-up of the two-level preconditioner on the small problem: a given basis of 32
        # vectors (the "simplified" reuse of another subset's basis) and one M_2l application.
        dict(name="coarse_small_fp64", kind="coarse", prec="fp64", nx=32, n_det=8, n_t=32768, block=4096, half_bw=512,
             n_bands=8, k=32, nrhs=1),
        # One product with A of the large mixed-precision problem (256x256, 128 detectors x 2^20 samples,
        # lambda 2048, 64 intervals): the call a solve of this size spends its time in.
        dict(name="A_large_mixed", kind="apply", prec="mixed", nx=256, n_det=128, n_t=1 << 20, block=16384, half_bw=2048,
             n_bands=128, nrhs=1, ragged=False, flagged=0.0),
        # A middle-sized scan as data cuts leave it: blocks of uneven, odd lengths and 1 % flagged samples.
        dict(name="A_ragged_mixed", kind="apply", prec="mixed", nx=64, n_det=24, n_t=180007, block=6000, half_bw=301,
             n_bands=24, nrhs=1, ragged=True, flagged=0.01),
        # A narrow noise band (lambda 16) on a serving-sized scan: the direct band filter.
        dict(name="A_narrow_mixed", kind="apply", prec="mixed", nx=128, n_det=64, n_t=1 << 19, block=16384, half_bw=16,
             n_bands=4, nrhs=1, ragged=False, flagged=0.0),
        # Right-hand side b = P^T W d of a serving-sized scan (float64-accurate products from float32 data).
        dict(name="rhs_mixed", kind="rhs", prec="mixed", nx=128, n_det=64, n_t=1 << 19, block=16384, half_bw=512,
             n_bands=4, nrhs=1, ragged=False, flagged=0.0),
        # Template-filtered product of the paper's ground-based pipeline: differenced timelines (Q, U),
        # first-order subscan polynomials and azimuth bins, double-float products.
        dict(name="A_templates_fp64", kind="templates", prec="fp64", products64=2, nx=256, n_det=32, n_t=1 << 20,
             block=16384, order=1, ground=True, stokes=1, nrhs=1),
        # Two-level preconditioner on a Monte Carlo batch: 512x512 patch, 64 coarse vectors, 64 maps.
        dict(name="M2l_batch", kind="precond", prec="fp64", nx=512, n_det=16, n_t=1 << 18, block=65536, half_bw=16,
             n_bands=16, k=64, nrhs=64),
        # A scan new to a server: pointing and weights set up from device arrays, M_BD, and the first
        # product with A and with M_BD.
        dict(name="new_scan_mixed", kind="setup", prec="mixed", nx=128, n_det=64, n_t=1 << 19, block=16384, half_bw=512,
             n_bands=4, nrhs=1),
        # The headline map: large scan, two-level preconditioner with 32 vectors from another realisation's
        # M_BD run, mixed precision, solved as tightly as the parity checks solve theirs.
        dict(name="solve_large_2l", kind="solve", prec="mixed", nx=256, n_det=128, n_t=1 << 20, block=16384, half_bw=2048,
             n_bands=128, nrhs=1, uneven=False, two_level=True, tol=1e-11, max_iter=500, products=100, graphs=False),
        # Monte Carlo batch: 64 maps of uneven length on one 32x32 master scan, captured iterations.
        dict(name="solve_mc_batch", kind="solve", prec="mixed", nx=32, n_det=8, n_t=1 << 20, block=4096, half_bw=512,
             n_bands=8, nrhs=64, uneven=True, two_level=False, tol=1e-11, max_iter=500, products=45, graphs=True),
    ]


def _logint(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["apply", "apply", "apply", "rhs", "templates", "precond", "setup", "solve", "coarse"])
    prec = rng.choice(["mixed", "fp64"])
    nx = _logint(rng, 16, 200)
    n_det = _logint(rng, 2, 64)
    block = rng.choice([4096, 8192, 16384, rng.randrange(1500, 20000)])
    # enough samples for every pixel, at most those of the largest case
    top = 6.0e7 if prec == "mixed" else 8.0e6
    n_t = max(_logint(rng, 1 << 15, 1 << 20), 12 * nx * nx // n_det)
    n_t = max(block, min(n_t, int(top / n_det)))
    if rng.random() < 0.6:
        n_t = max(1, n_t // block) * block
    half_bw = min(rng.choice([0, 16, _logint(rng, 4, 2048), _logint(rng, 128, 2048), 512]), block // 2)
    n_bands = rng.choice([1, min(4, n_det), n_det])
    c = dict(kind=kind, prec=prec, nx=nx, n_det=n_det, n_t=n_t, block=block, half_bw=half_bw, n_bands=n_bands, nrhs=1)
    if kind in ("apply", "rhs"):
        c.update(ragged=rng.random() < 0.4, flagged=rng.choice([0.0, 0.0, 0.01]))
        if n_det * n_t < 4_000_000:
            c.update(nrhs=rng.choice([1, 1, 2, 5, 16]))
    elif kind == "templates":
        c = dict(kind=kind, prec=prec, products64=rng.choice([1, 2]) if prec == "fp64" else 2, nx=nx, n_det=n_det,
                 n_t=n_t, block=block, order=rng.choice([-1, 0, 1, 1, 3]), ground=rng.random() < 0.7,
                 stokes=rng.choice([0, 1, 1, 2]), nrhs=1)
    elif kind == "precond":
        nx = _logint(rng, 24, 512)
        c = dict(kind=kind, prec=prec, nx=nx, n_det=16, n_t=max(1 << 14, nx * nx), block=max(1 << 14, nx * nx) // 4,
                 half_bw=16, n_bands=4, k=rng.choice([0, 8, 32, 64, 100]), nrhs=rng.choice([1, 1, 8, 33, 64]))
    elif kind == "coarse":
        c.update(prec="fp64", k=rng.choice([8, 25, 32]), n_t=max(block, min(n_t, 2_000_000 // n_det)))
    elif kind == "solve":
        c.update(n_t=max(block, min(n_t, (16_000_000 if prec == "mixed" else 1_500_000) // n_det)), uneven=False,
                 two_level=False, tol=1e-11, max_iter=500, products=50, graphs=False)
    return c


# ---------------- inputs ----------------

def _blocks(case):
    """Block offsets of the timeline: equal intervals, or uneven ones cut by `ragged`."""
    n_det, n_t, blk = case["n_det"], case["n_t"], case["block"]
    cuts = [0]
    r = np.random.default_rng(5)
    while cuts[-1] < n_t:
        step = int(r.integers(blk // 4, 2 * blk)) if case.get("ragged") else blk
        left = n_t - cuts[-1]
        cuts.append(cuts[-1] + (left if left < step + 32 else step))
    one = np.array(cuts, dtype=np.int64)
    off = np.concatenate([one[:-1] + d * n_t for d in range(n_det)] + [np.array([n_det * n_t])]).astype(np.int64)
    band = np.repeat(np.arange(n_det, dtype=np.int32) % case.get("n_bands", 1), len(one) - 1).astype(np.int32)
    return off, band


def _band(half_bw, f_knee):
    """c_0..c_lambda of the inverse of P(f) = 1 + f_knee / f, cut to |k| <= lambda and kept positive."""
    n = 16
    while n < 8 * max(1, half_bw):
        n *= 2
    f = np.fft.rfftfreq(n, 1.0 / FS_HZ)
    f[0] = f[1]
    c = np.fft.irfft(1.0 / (1.0 + f_knee / f), n=n)[:half_bw + 1].copy()
    if half_bw:
        grid = np.zeros(64 * n)
        grid[:half_bw + 1] = c
        grid[-half_bw:] = c[:0:-1]
        low = float(np.fft.rfft(grid).real.min())
        if low <= 0.0:
            c[0] += 1e-6 * c[0] - low
    return c


class _Scan:
    """Pointing on the device, blocks and bands on the host."""

    def __init__(self, case, seed):
        g = torch.Generator(device=DEV).manual_seed(seed)
        r = np.random.default_rng(seed)
        nx, n_det, n_t = case["nx"], case["n_det"], case["n_t"]
        self.nx, self.n_pix, self.n_det, self.n_t, self.n = nx, nx * nx, n_det, n_t, n_det * n_t
        self.block_off, self.block_band = _blocks(case)
        nb = int(self.block_band.max()) + 1
        self.f_knee = np.full(nb, 1.0) if nb <= 8 else r.uniform(0.1, 2.0, nb)
        if nb == 4:
            self.f_knee = np.array([0.1, 0.5, 1.0, 2.0])
        self.half_bw = case.get("half_bw", 0)
        self.band = np.stack([_band(self.half_bw, f) for f in self.f_knee])
        self.x0 = torch.from_numpy(r.uniform(0.0, 2.0 * nx, n_det)).to(DEV)
        y0 = float(r.uniform(0.0, nx))
        t = torch.arange(n_t, device=DEV, dtype=torch.float64)
        self.pix = torch.empty(self.n, device=DEV, dtype=torch.int32)
        for d in range(n_det):
            pos = torch.remainder(self.x0[d] + SPEED_PX * t, 2.0 * nx)
            ix = torch.minimum(pos, 2.0 * nx - pos).to(torch.int32).clamp_(0, nx - 1)
            iy = torch.remainder(y0 + d * nx / 4.0 / n_det + t * (nx / n_t), float(nx)).to(torch.int32).clamp_(0, nx - 1)
            self.pix[d * n_t:(d + 1) * n_t] = iy * nx + ix
        if case["kind"] == "templates":   # no half-wave plate: the detector's angle and a slow sky rotation
            rot = (math.pi / 4) * (t / n_t + float(r.uniform(0.0, 1.0)))
            det = (torch.arange(n_det, device=DEV, dtype=torch.float64) % 4) * (math.pi / 4)
            self.psi = torch.remainder(det[:, None] + rot[None, :], math.pi).reshape(-1).float()
        else:
            self.psi = torch.rand(self.n, generator=g, device=DEV) * math.pi
        self.psi.clamp_(max=float(np.nextafter(np.float32(np.pi), np.float32(0))))
        if case.get("flagged"):
            self.pix[torch.rand(self.n, generator=g, device=DEV) < case["flagged"]] = -1
        self.g = g

    def templates(self, case):
        """Subscans (sweeps between turnarounds, cut at block edges) and azimuth bins."""
        nx, n_t = self.nx, self.n_t
        t = torch.arange(n_t, device=DEV, dtype=torch.float64)
        cuts, az = [self.block_off], None
        bins = int(math.ceil(nx / AZ_BIN_PX))
        if case["ground"]:
            az = torch.empty(self.n, device=DEV, dtype=torch.int32)
        for d in range(self.n_det):
            raw = self.x0[d] + SPEED_PX * t
            sweep = torch.floor(raw / nx)
            turn = torch.nonzero(sweep[1:] != sweep[:-1]).reshape(-1) + 1
            cuts.append(turn.cpu().numpy().astype(np.int64) + d * n_t)
            if az is not None:
                pos = torch.remainder(raw, 2.0 * nx)
                pos = torch.minimum(pos, 2.0 * nx - pos)
                az[d * n_t:(d + 1) * n_t] = (pos / AZ_BIN_PX).to(torch.int32).clamp_(0, bins - 1)
        return np.unique(np.concatenate(cuts)), az, bins

    def map(self, nrhs):
        """Gaussian I/Q/U maps (sigma_I = 1, sigma_QU = 0.1)."""
        x = torch.randn((nrhs, self.n_pix, 3), generator=self.g, device=DEV, dtype=torch.float64)
        x[..., 1:] *= 0.1
        return x

    def tod(self, nrhs, dtype):
        """Timelines of a Gaussian sky plus 1/f noise (f_knee = 1 Hz), one after the other."""
        out = torch.empty((nrhs, self.n), device=DEV, dtype=dtype)
        ang = 2.0 * self.psi
        p = self.pix.clamp(min=0)
        ok = (self.pix >= 0).float()
        f = torch.fft.rfftfreq(4096, 1.0 / FS_HZ, device=DEV)
        f[0] = f[1]
        shape = torch.sqrt(1.0 + 1.0 / f)
        pad = -self.n % 4096
        for i in range(nrhs):
            sky = self.map(1)[0].float()
            w = torch.randn((self.n + pad) // 4096, 4096, generator=self.g, device=DEV)
            noise = torch.fft.irfft(torch.fft.rfft(w) * shape, n=4096).reshape(-1)[:self.n]
            sig = sky[:, 0][p] + sky[:, 1][p] * torch.cos(ang) + sky[:, 2][p] * torch.sin(ang)
            out[i] = noise + sig * ok
        return out


class _State:
    pass


def _context(case, sc, stream=None):
    ctx = M.Context(0, stream, M.MM_FP64 if case["prec"] == "fp64" else M.MM_FP32_MIXED)
    ctx.setup_pointing(sc.pix, sc.psi, sc.block_off, sc.block_band, sc.band, sc.n_pix, n_det=sc.n_det)
    return ctx


def _tod_dtype(case):
    return torch.float64 if case["prec"] == "fp64" else torch.float32


def _lengths(case, seed):
    if not case.get("uneven"):
        return None
    return np.random.default_rng(seed + 3).integers(case["n_t"] // 2, case["n_t"] + 1, case["nrhs"]).astype(np.int64)


def prepare(case, seed):
    s = _State()
    s.case, kind = case, case["kind"]
    sc = _Scan(case, seed)
    s.stream = torch.cuda.Stream() if case.get("graphs") else None
    if kind == "setup":
        s.scan = sc
        s.ctx = M.Context(0, None, M.MM_FP64 if case["prec"] == "fp64" else M.MM_FP32_MIXED)
        s.x = sc.map(case["nrhs"])
    else:
        torch.cuda.synchronize()
        s.ctx = _context(case, sc, s.stream.cuda_stream if s.stream else None)
    if kind == "templates":
        sub, az, bins = sc.templates(case)
        s.ctx.set_templates(case["order"], sub if case["order"] >= 0 else None, az, bins if case["ground"] else 0,
                            stokes=case["stokes"])
        if case["prec"] == "fp64":
            s.ctx.set_option("fp64_products", case["products64"])
    if kind in ("apply", "templates"):
        s.x = sc.map(case["nrhs"])
    elif kind == "rhs":
        s.d = sc.tod(case["nrhs"], _tod_dtype(case))
    elif kind in ("precond", "coarse"):
        s.ctx.build_bd(RCOND_MIN)
        s.Z = torch.randn((max(1, case["k"]), sc.n_pix, 3), generator=sc.g, device=DEV, dtype=torch.float64)
        s.x = torch.randn((case["nrhs"], sc.n_pix, 3), generator=sc.g, device=DEV, dtype=torch.float64)
        if kind == "precond":
            if case["k"]:
                torch.cuda.synchronize()
                s.ctx.set_coarse(s.Z)
            s.Z = None
    elif kind == "solve":
        s.ctx.build_bd(RCOND_MIN)
        s.d = sc.tod(case["nrhs"], _tod_dtype(case))
        s.lens = _lengths(case, seed)
        if case["graphs"]:
            s.ctx.set_option("graphs", 1)
        if case["two_level"]:
            other = sc.tod(1, _tod_dtype(case))
            torch.cuda.synchronize()
            s.ctx.set_option("harvest", 120)
            s.ctx.solve(other, M.MM_PRECOND_BD, tol=1e-8, max_iter=500)
            s.ctx.set_option("harvest", 0)
            s.ctx.build_coarse_from_solve(k=32)
            del other
    s.out = torch.empty((case["nrhs"], sc.n_pix, 3), device=DEV, dtype=torch.float64)
    torch.cuda.synchronize()
    return s


def run(s):
    case, ctx, kind = s.case, s.ctx, s.case["kind"]
    if kind in ("apply", "templates"):
        return ctx.apply_A(s.x, out=s.out)
    if kind == "rhs":
        return ctx.rhs(s.d, out=s.out)
    if kind == "precond":
        return ctx.apply_precond(M.MM_PRECOND_2L if case["k"] else M.MM_PRECOND_BD, s.x, out=s.out)
    if kind == "coarse":
        ctx.set_coarse(s.Z)
        return ctx.apply_precond(M.MM_PRECOND_2L, s.x, out=s.out)
    if kind == "setup":
        sc = s.scan
        ctx.setup_pointing(sc.pix, sc.psi, sc.block_off, sc.block_band, sc.band, sc.n_pix, n_det=sc.n_det)
        dropped = ctx.build_bd(RCOND_MIN)
        return {"dropped": dropped, "A": ctx.apply_A(s.x, out=s.out), "M": ctx.apply_precond(M.MM_PRECOND_BD, s.x)}
    m, info = ctx.solve(s.d, M.MM_PRECOND_2L if case["two_level"] else M.MM_PRECOND_BD, tol=case["tol"],
                        max_iter=case["max_iter"], rhs_len=s.lens, out=s.out)
    return list(m.unbind(0))


def work(case):
    n, n_pix, nrhs, kind = case["n_det"] * case["n_t"], case["nx"] ** 2, case["nrhs"], case["kind"]
    lam = case.get("half_bw", 0)
    maps = 2 * 24.0 * n_pix * nrhs
    # flops per sample of a product: pointing both ways, and the cheaper of the band sum and two real
    # transforms of a whole block with its spectrum
    span = min(case["block"], case["n_t"]) + lam
    fft = span / min(case["block"], case["n_t"]) * (5.0 * math.log2(max(2, span)) + 3.0)
    flt = 9.0 + min(2.0 * (2 * lam + 1), fft)
    elem = 8 if case["prec"] == "fp64" else 4
    product = dict(bytes=8.0 * n + maps, flops=flt * n * nrhs)
    if kind == "apply":
        return product
    if kind == "rhs":
        return dict(bytes=8.0 * n + elem * n * nrhs + maps / 2, flops=flt * n * nrhs)
    if kind == "templates":
        per = 9.0 + (8.0 * (case["order"] + 1) if case["order"] >= 0 else 0.0) * (2 if case["ground"] else 1) + 2.0
        return dict(bytes=(8.0 + (4.0 if case["ground"] else 0.0)) * n + maps, flops=per * n * nrhs)
    if kind == "precond":
        return dict(bytes=2 * 24.0 * n_pix * case["k"] + 48.0 * n_pix + maps,
                    flops=(6.0 * case["k"] * 3 + 15.0) * n_pix * nrhs)
    if kind == "coarse":
        k = case["k"]
        return dict(bytes=8.0 * n + 24.0 * n_pix * 3 * k, flops=flt * n * k + 4.0 * 3 * n_pix * k * k)
    if kind == "setup":
        return dict(bytes=8.0 * n + maps, flops=(flt + 15.0) * n)
    share = 0.75 if case["uneven"] else 1.0
    return dict(bytes=8.0 * n + elem * n * nrhs * share + maps / 2, flops=flt * n * nrhs * share * case["products"])


# ---------------- the same in 64 bits ----------------

class _Ref:
    """A = P^T W P, M_BD and the template filters in float64 with torch."""

    def __init__(self, sc, stokes=0):
        self.sc, self.stokes = sc, stokes
        self.p = sc.pix.long()
        ang = 2.0 * sc.psi.double()
        self.c, self.s = torch.cos(ang), torch.sin(ang)
        self.len = torch.from_numpy(np.diff(sc.block_off)).to(DEV)
        self.off = torch.from_numpy(sc.block_off[:-1]).to(DEV)
        self.bb = torch.from_numpy(sc.block_band.astype(np.int64)).to(DEV)
        self.nmax = int(self.len.max())
        self.uniform = bool((self.len == self.nmax).all())
        L = self.nmax + sc.half_bw
        while not self._smooth(L):
            L += 1
        self.L = L
        h = torch.zeros((sc.band.shape[0], L), device=DEV, dtype=torch.float64)
        b = torch.from_numpy(sc.band).to(DEV)
        h[:, :sc.half_bw + 1] = b
        if sc.half_bw:
            h[:, L - sc.half_bw:] = b[:, 1:].flip(1)
        self.H = torch.fft.rfft(h).real
        self.filter = self.weight

    @staticmethod
    def _smooth(n):
        for q in (2, 3, 5):
            while n % q == 0:
                n //= q
        return n == 1

    def weight(self, y):
        out = torch.empty_like(y)
        step = max(1, 120_000_000 // self.L)
        ar = torch.arange(self.nmax, device=DEV)
        for a in range(0, len(self.off), step):
            b = min(len(self.off), a + step)
            H = self.H[self.bb[a:b]]
            if self.uniform:
                lo, hi = a * self.nmax, b * self.nmax
                out[lo:hi] = torch.fft.irfft(torch.fft.rfft(y[lo:hi].view(b - a, -1), self.L) * H, self.L)[:, :self.nmax].reshape(-1)
            else:
                ok = ar[None, :] < self.len[a:b, None]
                at = (self.off[a:b, None] + ar[None, :])[ok]
                blk = torch.zeros((b - a, self.nmax), device=DEV, dtype=torch.float64)
                blk[ok] = y[at]
                out[at] = torch.fft.irfft(torch.fft.rfft(blk, self.L) * H, self.L)[:, :self.nmax][ok]
        return out

    def use_templates(self, order, sub, az, bins):
        n = self.sc.n
        wb = torch.from_numpy(self.sc.band[self.sc.block_band, 0]).to(DEV)
        block = torch.repeat_interleave(torch.arange(len(self.off), device=DEV), self.len)
        B = None
        if order >= 0:
            so = torch.from_numpy(sub).to(DEV)
            m = so[1:] - so[:-1]
            sid = torch.repeat_interleave(torch.arange(len(m), device=DEV), m)
            u = 2.0 * ((torch.arange(n, device=DEV) - so[sid]).double() + 0.5) / m[sid] - 1.0
            leg = [torch.ones_like(u), u, 1.5 * u * u - 0.5, (2.5 * u * u - 1.5) * u][:order + 1]
            for j in range(order + 1):   # a subscan of m samples carries m columns at most
                leg[j] = leg[j] * (m[sid] > j)
            B = torch.stack(leg, 1)
            G = torch.zeros((len(m), (order + 1) ** 2), device=DEV, dtype=torch.float64)
            G.index_add_(0, sid, (B[:, :, None] * B[:, None, :]).reshape(n, -1))
            G = G.view(len(m), order + 1, order + 1)
            ar = torch.arange(order + 1, device=DEV)
            G[:, ar, ar] += (m[:, None] <= ar[None, :]).double()
            Ginv = torch.linalg.inv(G)

        def poly(y):
            if B is None:
                return y
            mom = torch.zeros((len(m), order + 1), device=DEV, dtype=torch.float64)
            mom.index_add_(0, sid, B * y[:, None])
            coef = torch.einsum("sij,sj->si", Ginv, mom)
            return y - (B * coef[sid]).sum(1)

        if az is not None:
            key = block * bins + az.long()
            hits = torch.zeros(len(self.off) * bins, device=DEV, dtype=torch.float64)
            hits.index_add_(0, key, torch.ones(n, device=DEV, dtype=torch.float64))

        def f(y):
            y = poly(y)
            if az is not None:
                mean = torch.zeros_like(hits)
                mean.index_add_(0, key, y)
                y = poly(y - (mean / hits.clamp(min=1.0))[key])
            return wb[block] * y
        self.filter = f

    def project(self, x):
        v = x[self.p.clamp(min=0)]
        y = (v[:, 0] if self.stokes != 1 else 0.0) + (v[:, 1] * self.c + v[:, 2] * self.s if self.stokes != 2 else 0.0)
        return y * (self.p >= 0)

    def back(self, z):
        z = z * (self.p >= 0)
        p = self.p.clamp(min=0)
        out = torch.zeros((3, self.sc.n_pix), device=DEV, dtype=torch.float64)
        if self.stokes != 1:
            out[0].index_add_(0, p, z)
        if self.stokes != 2:
            out[1].index_add_(0, p, z * self.c)
            out[2].index_add_(0, p, z * self.s)
        return out.T.contiguous()

    def A(self, x):
        return self.back(self.filter(self.project(x)))

    def bd(self, select=True):
        """M_BD blocks, with badly observed pixels dropped from the pointing."""
        w0 = torch.repeat_interleave(torch.from_numpy(self.sc.band[self.sc.block_band, 0]).to(DEV), self.len)
        ok = (self.p >= 0).double()
        p = self.p.clamp(min=0)
        S = torch.zeros((7, self.sc.n_pix), device=DEV, dtype=torch.float64)
        c, s = self.c, self.s
        for i, v in enumerate((1.0, c, s, c * c, c * s, s * s)):
            S[i].index_add_(0, p, ok * w0 * v)
        S[6].index_add_(0, p, ok)
        m = torch.stack([S[0], S[1], S[2], S[1], S[3], S[4], S[2], S[4], S[5]], 1).view(-1, 3, 3)
        e = torch.linalg.eigvalsh(m.cpu()).to(DEV)
        rcond = e[:, 0] / e[:, 2].clamp(min=1e-300)
        if select:
            self.good = (S[6] >= 3) & (rcond >= RCOND_MIN)
            self.p = torch.where(self.good[p], self.p, torch.full_like(self.p, -1))
        else:   # a part of the scan: its selection is the whole scan's, pixels it does not see get no block
            self.good = self.good & (rcond > 1e-12)
        eye = torch.eye(3, device=DEV, dtype=torch.float64)
        self.M = torch.linalg.inv(torch.where(self.good[:, None, None], m, eye)) * self.good[:, None, None]
        return int((~self.good).sum())

    def precond(self, x):
        return torch.einsum("pij,pj->pi", self.M, x)

    def solve(self, d, tol=1e-14, most=400):
        b = self.back(self.filter(d))
        x, r = torch.zeros_like(b), b.clone()
        z = self.precond(r)
        p, rz, bn = z.clone(), (r * z).sum(), b.norm()
        for _ in range(most):
            q = self.A(p)
            al = rz / (p * q).sum()
            x += al * p
            r -= al * q
            if float(r.norm()) <= tol * float(bn):
                break
            z = self.precond(r)
            new = (r * z).sum()
            p = z + (new / rz) * p
            rz = new
        return x


def _prefix(sc, length):
    """The scan cut to the first `length` samples of every detector."""
    s = _State()
    s.__dict__.update(sc.__dict__)
    keep, off, band = [], [0], []
    for a, b, k in zip(sc.block_off[:-1], sc.block_off[1:], sc.block_band):
        d0 = a // sc.n_t * sc.n_t
        hi = min(b, d0 + length)
        if hi > a:
            off.append(off[-1] + hi - a)
            band.append(k)
    for d in range(sc.n_det):
        keep.append(torch.arange(d * sc.n_t, d * sc.n_t + length, device=DEV))
    keep = torch.cat(keep)
    s.pix, s.psi, s.n = sc.pix[keep], sc.psi[keep], len(keep)
    s.block_off, s.block_band = np.array(off, dtype=np.int64), np.array(band, dtype=np.int32)
    return s, keep


def exact(case, seed):
    kind, nrhs = case["kind"], case["nrhs"]
    sc = _Scan(case, seed)
    if kind == "templates":
        sub, az, bins = sc.templates(case)
        ref = _Ref(sc, case["stokes"])
        ref.use_templates(case["order"], sub, az, bins)
        return torch.stack([ref.A(x) for x in sc.map(nrhs)])
    ref = _Ref(sc)
    if kind == "apply":
        return torch.stack([ref.A(x) for x in sc.map(nrhs)])
    if kind == "rhs":
        return torch.stack([ref.back(ref.weight(d.double())) for d in sc.tod(nrhs, _tod_dtype(case))])
    if kind == "setup":
        x = sc.map(nrhs)
        dropped = ref.bd()
        return {"dropped": dropped, "A": torch.stack([ref.A(v) for v in x]), "M": torch.stack([ref.precond(v) for v in x])}
    if kind in ("precond", "coarse"):
        ref.bd()
        k = case["k"]
        Z = torch.randn((max(1, k), sc.n_pix, 3), generator=sc.g, device=DEV, dtype=torch.float64)
        X = torch.randn((nrhs, sc.n_pix, 3), generator=sc.g, device=DEV, dtype=torch.float64)
        if not k:
            return torch.stack([ref.precond(x) for x in X])
        AZ = torch.stack([ref.A(z) for z in Z])
        E = torch.einsum("apc,bpc->ab", Z, AZ)
        U = torch.linalg.solve(0.5 * (E + E.T).cpu(), torch.einsum("apc,rpc->ar", Z, X).cpu()).to(DEV)
        Y = X - torch.einsum("apc,ar->rpc", AZ, U)
        return torch.einsum("pij,rpj->rpi", ref.M, Y) + torch.einsum("apc,ar->rpc", Z, U)
    # solves: every map of a small batch, the first two of a large one
    ref.bd()
    d = sc.tod(nrhs, _tod_dtype(case))
    lens = _lengths(case, seed)
    if lens is None:
        return [ref.solve(d[i].double()) for i in range(nrhs)]
    got = []
    for i in range(nrhs):
        if i >= 2:
            got.append(None)
            continue
        part, keep = _prefix(sc, int(lens[i]))
        one = _Ref(part)
        one.good = ref.good
        one.p = ref.p[keep]
        one.bd(select=False)
        got.append(one.solve(d[i][keep].double()))
    return got
