"""The calls whose time matters to a user of this package, with their sizes.

A case names an operator form (``prec``: plain FP32, split BF16 on the tensor
cores, lateral FFT), what is called (``op``) and the sizes of the scan grid,
the volume, the signals and the slab window.  ``listed`` holds the fixed
cases, ``draw`` gives others of the same ranges, ``prepare`` makes a model and
inputs, ``run`` is one call as a program makes it, and ``exact`` evaluates the
same call in 64 bits from the definition of the model (Eqs. 1-4) with torch.

The sizes are those of the configurations: the 32x32x48 volume, the
200x200x300 volume (61x61 window), the batched and served reconstructions
(scans of 64 to 256 positions a side, 128 to 384 depths, 512 to 1024 samples,
focal lengths of 3 to 6 mm, apertures of 2 to 4 mm), and ragged sizes as the
tests use them.
"""
import math

import numpy as np
import torch

from paper_2009_10173_gb300 import binding as B
from paper_2009_10173_gb300 import configs
from paper_2009_10173_gb300.model import Model

PREC = {"fp32": B.OAM_PREC_FP32, "bf16x3": B.OAM_PREC_BF16X3, "fft": B.OAM_PREC_FFT}
C_MPS, FS, FC, BW, TRUNC = 1500.0, 250e6, 30e6, 1.0, 5.0
FILTER = dict(f_lo=0.5e6, f_hi=80e6, half=511)  # the band of the paper's second simulation
POWER_ITERS, LAMBDA_REL = 20, 1e-3


def _case(name, prec, op, base, **over):
    c = configs.scaled(base, **over)
    return dict(name=name, prec=prec, op=op, px=c["px"], py=c["py"], nz=c["nz"], nt=c["nt"], win=c["win"],
                dx_um=c["dx_m"] * 1e6, dz_um=c["dz_m"] * 1e6, z0_um=c["z0_rel_m"] * 1e6,
                focal_mm=c["focal_m"] * 1e3, aperture_mm=c["aperture_m"] * 1e3, patches=c["n_patches"])


def _scan(name, prec, op, scan, nz, nt, **over):
    """A job of the batched and served workloads: the volume is centred on the focus."""
    base = configs.VOLUME_200
    return _case(name, prec, op, base, px=scan, py=scan, nz=nz, nt=nt, z0_rel_m=-(nz / 2) * base["dz_m"], **over)


def listed():
    tiny, vol = configs.TINY_32, configs.VOLUME_200
    return [
        # the smallest volume: one forward projection, as an interactive preview or a test makes it
        _case("fp32_forward_tiny", "fp32", "forward", tiny),
        # the small reconstruction of the tests and demos: ten LSQR iterations in one call
        _case("fp32_lsqr10_tiny", "fp32", "lsqr10", tiny),
        # ragged sizes: no dimension fits a tile
        _case("fp32_adjoint_ragged", "fp32", "adjoint", tiny, px=70, py=37, nz=52, nt=200, win=15, n_patches=800,
              dz_m=8e-6, z0_rel_m=-200e-6),
        # the plain form at the paper's volume size: the largest single call
        _case("fp32_forward_volume", "fp32", "forward", vol),
        # the tensor-core form at that size, both directions: the solvers call these ~100 to ~250 times a volume
        _case("bf16x3_forward_volume", "bf16x3", "forward", vol),
        _case("bf16x3_adjoint_volume", "bf16x3", "adjoint", vol),
        # the tensor-core form on a small job of a batch
        _scan("bf16x3_forward_scan96", "bf16x3", "forward", 96, 192, 768),
        # the lateral-FFT form: the paper's volume, the largest and the smallest scan of a batch
        _case("fft_forward_volume", "fft", "forward", vol),
        _scan("fft_adjoint_scan256", "fft", "adjoint", 256, 384, 1024),
        _scan("fft_forward_scan64", "fft", "forward", 64, 128, 512),
        # one served request: build its model, MB-L2 (LSQR-30) and MB-L1 (FISTA-50), release the model
        _scan("fft_request_scan128", "fft", "request", 128, 192, 768, focal_m=5e-3),
        # band-pass filtering of measured signals before a reconstruction
        _case("filter_volume", "fft", "filter", vol),
    ]


def draw(rng):
    def logint(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    while True:
        prec = rng.choice(["fp32", "bf16x3", "fft", "bf16x3", "fft"])
        op = rng.choice(["forward", "adjoint", "forward", "adjoint", "lsqr10" if prec != "bf16x3" else "adjoint",
                         "filter" if prec == "fft" else "forward", "request" if prec == "fft" else "adjoint"])
        side = logint(24, 256)
        px, py = side, max(16, min(256, int(side * rng.uniform(0.6, 1.4))))
        if rng.random() < 0.3:
            px, py = rng.choice(configs.BATCH_SCAN), rng.choice(configs.BATCH_SCAN)
        nz = logint(32, 384)
        win = min(61, 2 * logint(4, 31) - 1)
        dz = 5.0
        c = dict(prec=prec, op=op, px=px, py=py, nz=nz, nt=4 * rng.randrange(48, 257), win=win, dx_um=10.0, dz_um=dz,
                 z0_um=-(nz / 2) * dz, focal_mm=round(rng.uniform(3.0, 6.0), 3),
                 aperture_mm=round(rng.uniform(2.0, 4.0), 3), patches=8 * rng.randrange(100, 251))
        n_lo, n_hi, _, cost = _bands(c)
        if n_hi + 8 > 1024 or n_hi - n_lo > 416 or nz > 384:
            continue  # more samples than a batch's largest count, or wider than the tensor cores' accumulator
        c["nt"] = max(c["nt"], (n_hi + 8 + 3) // 4 * 4)
        work = {"fp32": 1.0, "bf16x3": 1 / 60.0, "fft": 1 / 700.0}[prec] * px * py * cost
        if op in ("lsqr10", "request"):
            work *= {"lsqr10": 21, "request": 200}[op]
        if work > 200 * 200 * _bands(listed()[3])[3]:
            continue  # costs more than the largest listed case
        return c


# ------------------------------------------------------------------ inputs
def _cfg(case):
    return dict(focal_m=case["focal_mm"] * 1e-3, aperture_m=case["aperture_mm"] * 1e-3, hole_m=0.0, c_mps=C_MPS,
                n_patches=case["patches"], fc_hz=FC, frac_bw=BW, trunc_sigma=TRUNC, px=case["px"], py=case["py"],
                nz=case["nz"], nt=case["nt"], win=case["win"], dx_m=case["dx_um"] * 1e-6, dy_m=case["dx_um"] * 1e-6,
                dz_m=case["dz_um"] * 1e-6, z0_rel_m=case["z0_um"] * 1e-6, fs_hz=FS, t0_s=float("nan"))


def _volume(case, seed):
    """Absorbed energy: round absorbers of 20 to 50 um and straight tubes of 5 to 30 um radius on a zero background."""
    g = _cfg(case)
    r = np.random.Generator(np.random.PCG64(seed))
    f32 = dict(dtype=torch.float32, device="cuda")
    y = torch.arange(g["py"], **f32)[:, None, None] * (g["dy_m"] * 1e6)
    x = torch.arange(g["px"], **f32)[None, :, None] * (g["dx_m"] * 1e6)
    z = torch.arange(g["nz"], **f32)[None, None, :] * (g["dz_m"] * 1e6)
    ext = np.array([g["py"] * g["dy_m"], g["px"] * g["dx_m"], g["nz"] * g["dz_m"]]) * 1e6
    H = torch.zeros((g["py"], g["px"], g["nz"]), **f32)
    for _ in range(30):
        c, D, a = r.uniform(0, 1, 3) * ext, r.uniform(20, 50), r.uniform(0.5, 1.0)
        d2 = (y - c[0]) ** 2 + (x - c[1]) ** 2 + (z - c[2]) ** 2
        H = torch.maximum(H, torch.where(d2 < 2.25 * D * D, a * torch.exp(-4 * math.log(2.0) / (D * D) * d2), 0.0))
    for _ in range(8):
        p, q, rad = r.uniform(0, 1, 3) * ext, r.uniform(0, 1, 3) * ext, r.uniform(5, 30)
        u = (q - p) / np.linalg.norm(q - p)
        dy, dx, dz = y - p[0], x - p[1], z - p[2]
        t = dy * u[0] + dx * u[1] + dz * u[2]
        H = torch.maximum(H, (dy * dy + dx * dx + dz * dz - t * t <= rad * rad).float())
    return H.contiguous()


def _signals(case, seed):
    """Measured A-lines: arrivals of point absorbers that spread with defocus, and white noise at 20 dB."""
    g = _cfg(case)
    r = np.random.Generator(np.random.PCG64(seed))
    gen = torch.Generator(device="cuda").manual_seed(seed)
    f32 = dict(dtype=torch.float32, device="cuda")
    sigma = FS / (2 * math.pi * FC * BW / (2 * math.sqrt(2 * math.log(2.0))))
    n_lo, _, g0, _ = _bands(case)
    n = torch.arange(g["nt"], **f32)
    y, x = torch.arange(g["py"], **f32) * g["dy_m"], torch.arange(g["px"], **f32) * g["dx_m"]
    na = 0.5 * g["aperture_m"] / g["focal_m"]
    s = torch.zeros((g["py"], g["px"], g["nt"]), **f32)
    for _ in range(24):
        yc, xc = r.uniform(0, g["py"] * g["dy_m"]), r.uniform(0, g["px"] * g["dx_m"])
        zc = g["z0_rel_m"] + r.uniform(0.05, 0.95) * g["nz"] * g["dz_m"]
        w = 20e-6 + 0.7 * na * abs(zc)
        rho2 = (y - yc)[:, None] ** 2 + (x - xc)[None, :] ** 2
        iy = torch.nonzero((y - yc).abs() < 3 * w).flatten()
        ix = torch.nonzero((x - xc).abs() < 3 * w).flatten()
        if not len(iy) or not len(ix):
            continue
        ys, xs = slice(int(iy[0]), int(iy[-1]) + 1), slice(int(ix[0]), int(ix[-1]) + 1)
        q = rho2[ys, xs]
        tau = n - (g0 + FS / C_MPS * (zc + math.copysign(0.5, zc) * q / (abs(zc) + 100e-6)))[..., None]
        e = torch.exp(-tau * tau / (2 * sigma * sigma))
        om = 2 * math.pi * FC / FS
        s[ys, xs] += float(r.uniform(0.5, 1.0)) * torch.exp(-q / (w * w))[..., None] * \
            (-e * (tau / (sigma * sigma) * torch.cos(om * tau) + om * torch.sin(om * tau)))
    rms = float(s.double().pow(2).mean().sqrt())
    s += (0.1 * rms if rms > 0 else 1.0) * torch.randn(s.shape, generator=gen, **f32)
    return s


def _input(case, seed):
    return _volume(case, seed) if case["op"] == "forward" else _signals(case, seed)


def prepare(case, seed):
    state = {"op": case["op"], "x": _input(case, seed), "cfg": _cfg(case), "prec": PREC[case["prec"]]}
    if case["op"] != "request":
        state["model"] = Model(state["cfg"], precision=state["prec"])
        if case["op"] == "filter":
            state["model"].set_filter(B.oam_bandpass_taps(FILTER["f_lo"], FILTER["f_hi"], FS, FILTER["half"]))
    return state


def run(state):
    op, x = state["op"], state["x"]
    if op == "request":
        m = Model(state["cfg"], precision=state["prec"])
        l2, _ = m.lsqr(x, 30, want_info=False)
        l1, _ = m.fista(x, 50, power_iters=POWER_ITERS, lambda_rel=LAMBDA_REL, want_info=False)
        m.close()
        return {"l2": l2, "l1": l1}
    m = state["model"]
    if op == "forward":
        return m.forward(x)
    if op == "adjoint":
        return m.adjoint(x)
    if op == "filter":
        return m.filter_signals(x)
    return m.lsqr(x, 10, want_info=False)[0]


# ------------------------------------------------------------------ least work
def _bands(case):
    """Support [n_lo, n_hi) of the slab in samples, the sample of a focal arrival, and the slab entries over all taps.

    From the distances of the sensor's axis and rim (the extremes of each ring lie in and against the voxel's azimuth).
    """
    g = _cfg(case)
    F, R = g["focal_m"], (g["win"] - 1) // 2
    sigma = FS / (2 * math.pi * FC * BW / (2 * math.sqrt(2 * math.log(2.0))))
    th = np.linspace(0.0, math.asin(0.5 * g["aperture_m"] / F), 9)
    th = np.concatenate([-th[1:], th])
    a = np.arange(R + 1)
    rho = np.sqrt(a[:, None] ** 2.0 + a[None, :] ** 2) * g["dx_m"]
    z = g["z0_rel_m"] + np.arange(g["nz"]) * g["dz_m"]
    rn = z[None, None, :, None] * np.cos(th) + rho[..., None, None] * np.sin(th)
    num = 2 * F * rn + (rho[..., None] ** 2 + z ** 2)[..., None]
    dd = num / (np.sqrt(F * F + num) + F) * FS / C_MPS
    lo, hi = dd.min(axis=-1), dd.max(axis=-1)
    g0 = FS * F / C_MPS - (math.floor(FS * F / C_MPS + lo.min() - TRUNC * sigma) - 2)
    band = hi - lo + 2 * TRUNC * sigma
    mult = np.where(a == 0, 1, 2)
    entries = float((mult[:, None, None] * mult[None, :, None] * band).sum())
    n_lo = int(math.floor(g0 + lo.min() - TRUNC * sigma))
    return n_lo, int(math.ceil(g0 + hi.max() + TRUNC * sigma)) + 1, g0, entries


def work(case):
    """Input and output once, the slab's distinct entries once per operator; the flops are those of the transforms and
    the products of the lateral spectrum, the least that is known for these correlations."""
    px, py, nz, nt, R = case["px"], case["py"], case["nz"], case["nt"], (case["win"] - 1) // 2
    vol, sig = 4.0 * px * py * nz, 4.0 * px * py * nt
    n_lo, n_hi, _, entries = _bands(case)
    if case["op"] == "filter":
        n = nt + FILTER["half"]
        return {"bytes": 2 * sig, "flops": px * py * (5.0 * n * math.log2(n) + n)}
    slab = 4.0 * entries / 7.5  # one of each eight mirrored and transposed taps (fewer on the axes)
    ny, nx, chan = py + R, px + R, nz + n_hi - n_lo
    per_tap = entries / case["win"] ** 2
    flops = 2.5 * ny * nx * math.log2(ny * nx) * chan + 2.0 * ny * nx * per_tap
    one = vol + sig + slab
    if case["op"] in ("forward", "adjoint"):
        return {"bytes": one, "flops": flops}
    ops = 21 if case["op"] == "lsqr10" else 61 + 2 * POWER_ITERS + 1 + 100
    return {"bytes": ops * one, "flops": ops * flops}


# ------------------------------------------------------------------ 64 bits
class _Exact:
    """The operators of the definition in 64 bits: the slab as the sum over the sensor's patches, applied as a product
    of zero-padded lateral spectra."""

    def __init__(self, case):
        self.g = g = _cfg(case)
        self.f64 = dict(dtype=torch.float64, device="cuda")
        F, M, R = g["focal_m"], g["n_patches"], (g["win"] - 1) // 2
        self.R = R
        sigma = FS / (2 * math.pi * FC * BW / (2 * math.sqrt(2 * math.log(2.0))))
        om, cut = 2 * math.pi * FC / FS, TRUNC * sigma
        # rings uniform in polar angle, 8 u_r patches each, the units after the first by ring area (largest remainder)
        th_out = math.asin(g["aperture_m"] / (2 * F))
        cap = 2 * math.pi * F * F * (1 - math.cos(th_out))
        units = M // 8
        v = th_out * F * math.sqrt(M / cap)
        rings = max(1, min(int(math.floor(v + 0.5)), units))
        edge = np.cos(np.linspace(0.0, th_out, rings + 1))
        area = 2 * math.pi * F * F * (edge[:-1] - edge[1:])
        share = (units - rings) * area / cap
        u = 1 + np.floor(share).astype(int)
        order = np.argsort(-(share - np.floor(share)), kind="stable")
        u[order[:units - u.sum()]] += 1
        mid = 0.5 * (edge[:-1] + edge[1:])
        nrm, wts = [], []
        for c, ar, n in zip(mid, area, 8 * u):
            phi = 2 * math.pi * (np.arange(n) + 0.5) / n
            sn = math.sqrt(1 - c * c)
            nrm.append(np.stack([sn * np.cos(phi), sn * np.sin(phi), np.full(n, c)], axis=1))
            wts.append(np.full(n, ar / n * 1e6))
        nrm = torch.tensor(np.concatenate(nrm), **self.f64)
        wts = torch.tensor(np.concatenate(wts), **self.f64)
        pairs = [(b, a) for b in range(R + 1) for a in range(b, R + 1)]
        idx = np.zeros((2 * R + 1, 2 * R + 1), dtype=np.int64)
        where = {p: i for i, p in enumerate(pairs)}
        for b in range(-R, R + 1):
            for a in range(-R, R + 1):
                idx[b + R, a + R] = where[tuple(sorted((abs(b), abs(a))))]
        self.idx = torch.tensor(idx, device="cuda")
        off = torch.tensor(pairs, **self.f64) * g["dx_m"]

        def delta(k):
            z = g["z0_rel_m"] + k * g["dz_m"]
            rn = off[:, 1:2] * nrm[:, 0] + off[:, 0:1] * nrm[:, 1] + z * nrm[:, 2]
            num = 2 * F * rn + (off ** 2).sum(1, keepdim=True) + z * z
            return num / (torch.sqrt(F * F + num) + F)

        dmin = min(float(delta(k).min()) for k in range(g["nz"]))
        n0 = math.floor(FS / C_MPS * (F + dmin) - TRUNC * sigma) - 2
        G = FS * F / C_MPS - n0
        T = int(math.ceil(cut)) + 1
        t = torch.arange(-T, T + 1, **self.f64)
        self.band, self.spec = [], []
        self.P = 2
        need = max(g["px"], g["py"]) + R
        while True:
            m = self.P
            for p in (2, 3, 5):
                while m % p == 0:
                    m //= p
            if m == 1 and self.P >= need:
                break
            self.P += 1
        for k in range(g["nz"]):
            dd = delta(k)
            D = FS / C_MPS * dd + G
            ref = torch.round(D)
            lo = int(ref.min()) - T
            width = int(ref.max()) + T + 1 - lo
            out = torch.zeros(len(pairs) * width, **self.f64)
            step = max(1, (1 << 24) // (len(pairs) * len(t)))
            for j in range(0, M, step):
                f = (D[:, j:j + step] - ref[:, j:j + step])[..., None]
                tau = t - f
                val = -torch.exp(-tau * tau / (2 * sigma * sigma)) * \
                    (tau / (sigma * sigma) * torch.cos(om * tau) + om * torch.sin(om * tau))
                val = torch.where(tau.abs() <= cut, val, 0.0) * \
                    (wts[j:j + step] / ((F + dd[:, j:j + step]) * 1e3))[..., None]
                at = (ref[:, j:j + step, None] + t - lo).long() + \
                    width * torch.arange(len(pairs), device="cuda")[:, None, None]
                out.index_add_(0, at.flatten(), val.flatten())
            b0, b1 = max(0, -lo), min(width, g["nt"] - lo)
            self.band.append((lo + b0, lo + b1))
            self.spec.append(out.view(len(pairs), width)[:, b0:b1])

    def _hat(self, k, cache):
        """Real lateral spectrum of depth k's slab, [P, P/2 + 1, samples]."""
        s = self.spec[k]
        if s.dim() == 3:
            return s
        R, W = self.R, 2 * self.R + 1
        full = torch.zeros((self.P, self.P, s.shape[1]), **self.f64)
        r = (torch.arange(W, device="cuda") - R) % self.P
        full[r[:, None], r[None, :]] = s[self.idx]
        h = torch.fft.rfft2(full, dim=(0, 1)).real.contiguous()
        if cache:
            self.spec[k] = h
        return h

    def forward(self, H, cache=False):
        g, P = self.g, self.P
        Hf = torch.fft.rfft2(H, s=(P, P), dim=(0, 1))
        acc = torch.zeros((P, P // 2 + 1, g["nt"]), dtype=torch.complex128, device="cuda")
        for k, (a, b) in enumerate(self.band):
            acc[:, :, a:b] += self._hat(k, cache) * Hf[:, :, k:k + 1]
        return torch.fft.irfft2(acc, s=(P, P), dim=(0, 1))[:g["py"], :g["px"]].contiguous()

    def adjoint(self, s, cache=False):
        g, P = self.g, self.P
        sf = torch.fft.rfft2(s, s=(P, P), dim=(0, 1))
        out = torch.empty((P, P // 2 + 1, g["nz"]), dtype=torch.complex128, device="cuda")
        for k, (a, b) in enumerate(self.band):
            out[:, :, k] = (self._hat(k, cache) * sf[:, :, a:b]).sum(-1)
        return torch.fft.irfft2(out, s=(P, P), dim=(0, 1))[:g["py"], :g["px"]].contiguous()

    def lsqr(self, s, iters):
        """LSQR (Paige and Saunders) without damping, from zero."""
        beta = s.norm()
        u = s / beta
        v = self.adjoint(u, True)
        alpha = v.norm()
        v = v / alpha
        w, x = v.clone(), torch.zeros_like(v)
        phibar, rhobar = beta, alpha
        for _ in range(iters):
            u = self.forward(v, True) - alpha * u
            beta = u.norm()
            u = u / beta
            v = self.adjoint(u, True) - beta * v
            alpha = v.norm()
            v = v / alpha
            rho = torch.sqrt(rhobar * rhobar + beta * beta)
            c, sn = rhobar / rho, beta / rho
            theta, rhobar, phi, phibar = sn * alpha, -c * alpha, c * phibar, sn * phibar
            x = x + phi / rho * w
            w = v - theta / rho * w
        return x

    def fista(self, s, iters):
        """Non-negative FISTA of ||s - A H||^2 + lambda ||H||_1 with the step from a power iteration."""
        v = torch.ones((self.g["py"], self.g["px"], self.g["nz"]), **self.f64)
        for _ in range(POWER_ITERS):
            th = self.adjoint(self.forward(v, True), True)
            mu = th.norm() / v.norm()
            v = th / th.norm()
        L = 2 * 1.01 * mu
        lam = LAMBDA_REL * self.adjoint(s, True).abs().max()
        x = torch.zeros_like(v)
        y, t = x, 1.0
        for _ in range(iters):
            z = y - 2.0 / L * self.adjoint(self.forward(y, True) - s, True)
            xn = torch.clamp(z - lam / L, min=0.0)
            tn = 0.5 * (1 + math.sqrt(1 + 4 * t * t))
            y = xn + (t - 1) / tn * (xn - x)
            x, t = xn, tn
        return x


def exact(case, seed):
    x = _input(case, seed).double()
    if case["op"] == "filter":
        L = FILTER["half"]
        m = torch.arange(-L, L + 1, dtype=torch.float64, device="cuda")
        w = 0.42 + 0.5 * torch.cos(math.pi * m / (L + 1)) + 0.08 * torch.cos(2 * math.pi * m / (L + 1))
        hi, lo = 2 * FILTER["f_hi"] / FS, 2 * FILTER["f_lo"] / FS
        h = w * (hi * torch.sinc(hi * m) - lo * torch.sinc(lo * m))
        n = x.shape[-1] + 2 * L
        hf = torch.fft.rfft(h, n=n)
        return torch.cat([torch.fft.irfft(torch.fft.rfft(r, n=n) * hf, n=n)[..., L:L + x.shape[-1]]
                          for r in x.split(16)])
    e = _Exact(case)
    if case["op"] == "forward":
        return e.forward(x)
    if case["op"] == "adjoint":
        return e.adjoint(x)
    if case["op"] == "lsqr10":
        return e.lsqr(x, 10)
    return {"l2": e.lsqr(x, 30), "l1": e.fista(x, 50)}
