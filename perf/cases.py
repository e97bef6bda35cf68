"""The work whose speed is followed: passes of the estimator as a program makes them, through `Plan`, `Batch` and
`modal_fnl`, from one small map to high-resolution batches.

A case is a dict of plain values:
  kind    what the pass does (see `run`)
  lmax, P, nrings, nphi, prec     the plan
  maps    maps in the batch
  linear  Monte Carlo pair means of the linear term: "none", "pixel" or "ring"
  sims    simulations behind those means
  mask    "none", "band" (the 20-degree band of rings) or "holes" (a band and round holes, per pixel)

Inputs are Gaussian a_lm with C_l = 1 / (l (l + 1)), white noise maps, and modal coefficients with a well-conditioned
covariance; all made on the GPU from the seed.
"""
import math

import numpy as np
import torch

import paper_1105_2791_gb300 as M

TWO_PI = 2.0 * math.pi


def _case(name, kind, lmax, P, nrings, nphi, prec, maps, linear="none", sims=0, mask="none"):
    return {"name": name, "kind": kind, "lmax": lmax, "P": P, "nrings": nrings, "nphi": nphi, "prec": prec,
            "maps": maps, "linear": linear, "sims": sims, "mask": mask}


def listed():
    return [
        # one small map at the default precision: launches and latency, as in a test or a parameter scan
        _case("beta_l32", "beta", 32, 6, 33, 128, "fp32", 1, "pixel", 32),
        # a batch of Monte Carlo maps at WMAP resolution, masked: the bulk of a covariance run
        _case("beta_l500", "beta", 500, 10, 501, 1024, "fp16x3", 64, "pixel", 32, "band"),
        # high resolution with 816 modes: the headline coefficient pass
        _case("beta_l2000", "beta", 2000, 16, 2001, 4096, "fp16x3", 12, "pixel", 12, "band"),
        # the default precision on a ragged grid with a pixel mask, a batch that is no multiple of anything
        _case("beta_l250_fp32", "beta", 250, 8, 273, 512, "fp32", 21, "pixel", 16, "holes"),
        # the Monte Carlo pair means of the linear term from a batch of simulations
        _case("means_l500", "means", 500, 10, 501, 1024, "fp16x3", 64, "pixel", 0, "band"),
        # the gradient of a weighted sum of coefficients (the adjoint workload)
        _case("grad_l1000", "grad", 1000, 12, 1001, 2048, "fp16x3", 16, "pixel", 16, "band"),
        # filtered maps alone, odd sizes, the other accurate tensor-core precision
        _case("maps_l767", "maps", 767, 7, 801, 2048, "3xtf32", 5),
        # noise maps to a_lm: the quadrature analysis that precedes a noisy simulation
        _case("alm_l1000", "alm", 1000, 12, 1001, 2048, "fp16x3", 32),
        # trispectrum modes with the Monte Carlo terms per ring
        _case("tau_l300", "tau", 300, 10, 301, 1024, "fp16x3", 8, "ring", 16, "band"),
        # the estimate: covariance of 816 modes factored, f_NL of a batch and its weights
        _case("solve_816", "solve", 64, 16, 65, 256, "fp16x3", 32),
        # coefficient passes of three resolutions as one batch
        _case("batch_l125_250_500", "batch", 500, 12, 501, 1024, "fp16x3", 16, "pixel", 16, "band"),
        # f_NL of a batch and its gradient through autograd, default precision
        _case("fnl_l200_fp32", "fnl", 200, 6, 201, 512, "fp32", 16, "pixel", 16, "none"),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["beta", "beta", "beta", "means", "grad", "grad", "maps", "alm", "tau", "solve", "batch", "fnl"])
    prec = rng.choice(["fp16x3", "fp16x3", "fp32", "fp32", "3xtf32"])
    lmax = _log_int(rng, 24, 1400 if prec != "fp32" else 600)
    P = rng.randint(3, 16)
    linear, sims, mask = "none", 0, rng.choice(["none", "band", "holes"])
    if kind == "solve":
        lmax = 32
    if kind in ("tau", "fnl"):
        lmax, P = _log_int(rng, 24, 300), rng.randint(3, 10 if kind == "tau" else 8)
    if kind == "batch":
        lmax, P = _log_int(rng, 64, 500), rng.randint(4, 12)
    nrings = lmax + 1 + rng.randint(0, max(1, lmax // 8))
    nphi = 16
    while nphi < 2 * lmax + 2:
        nphi *= 2
    if kind in ("beta", "grad", "tau", "batch", "fnl") and rng.random() < 0.8:
        linear, sims = "pixel" if mask == "holes" or rng.random() < 0.7 else "ring", rng.randint(4, 16)
    if kind == "means":
        linear = "pixel"
    # as many maps as keep maps x modes x pixels within a quarter of the largest listed case
    most = int(max(1, min(64, 4e8 / (nrings * nphi * P))))
    maps = _log_int(rng, 1, most)
    return {"kind": kind, "lmax": lmax, "P": P, "nrings": nrings, "nphi": nphi, "prec": prec, "maps": maps,
            "linear": linear, "sims": sims, "mask": mask}


# ------------------------------------------------------------------ sizes and inputs

def _n_alm(lmax):
    return (lmax + 1) * (lmax + 2) // 2


def _n_modes(P):
    return P * (P + 1) * (P + 2) // 6


def _cl(lmax):
    cl = np.zeros(lmax + 1)
    l = np.arange(2, lmax + 1, dtype=float)
    cl[2:] = 1.0 / (l * (l + 1.0))
    return cl


def _basis(lmax, P):
    x = 2.0 * np.arange(lmax + 1) / max(lmax, 1) - 1.0
    return np.stack([np.polynomial.legendre.legval(x, np.eye(P)[p]) for p in range(P)])


def _lm(lmax):
    """(l, m) of the packed m-major order, on the GPU."""
    m = torch.repeat_interleave(torch.arange(lmax + 1, device="cuda"),
                                torch.arange(lmax + 1, 0, -1, device="cuda"))
    start = m * (2 * lmax + 3 - m) // 2
    return m + torch.arange(m.numel(), device="cuda") - start, m


def _gen(seed, stream):
    return torch.Generator(device="cuda").manual_seed(int(seed) * 16 + stream)


def _alm(lmax, n, seed, stream):
    """Gaussian a_lm, complex64 [n][n_alm]; a_l0 real."""
    l, m = _lm(lmax)
    s = torch.sqrt(torch.from_numpy(_cl(lmax)).cuda()[l])
    z = torch.randn((n, l.numel(), 2), generator=_gen(seed, stream), device="cuda", dtype=torch.float32)
    re = torch.where(m == 0, s, s * math.sqrt(0.5)).float()
    im = torch.where(m == 0, torch.zeros_like(s), s * math.sqrt(0.5)).float()
    return torch.complex(z[..., 0] * re, z[..., 1] * im).contiguous()


def _mask(c, lmax=None, nrings=None, nphi=None):
    """(ring_mask or None, pix_mask or None) as float32 arrays."""
    nrings, nphi = nrings or c["nrings"], nphi or c["nphi"]
    if c["mask"] == "none":
        return None, None
    th = np.pi * (np.arange(nrings) + 0.5) / nrings          # close to the ring colatitudes
    band = (np.abs(np.cos(th)) >= math.sin(math.radians(20.0))).astype(np.float32)
    if c["mask"] == "band":
        return band, None
    phi = TWO_PI * np.arange(nphi) / nphi
    pm = np.repeat(band[:, None], nphi, axis=1)
    for t0, p0, r in ((0.5, 1.0, 0.1), (0.9, 4.0, 0.05), (2.4, 2.0, 0.15), (2.7, 5.5, 0.08)):
        cosd = np.cos(th)[:, None] * math.cos(t0) + np.sin(th)[:, None] * math.sin(t0) * np.cos(phi[None, :] - p0)
        pm[cosd > math.cos(r)] = 0.0
    return None, pm


def _betas(n, count, seed, stream):
    """Modal coefficients with a well-conditioned covariance (an orthonormalised mode set), float64 [count][n]."""
    mix = torch.randn((n, n), generator=_gen(0, 15), device="cuda", dtype=torch.float64) * (0.3 / math.sqrt(n))
    mix += torch.eye(n, device="cuda", dtype=torch.float64)
    return torch.randn((count, n), generator=_gen(seed, stream), device="cuda", dtype=torch.float64) @ mix.T


def _alpha(n, seed):
    return torch.randn(n, generator=_gen(seed, 9), device="cuda", dtype=torch.float64).cpu().numpy()


def _batch_parts(c):
    """The plans of a mixed batch: lmax / 4, lmax / 2 and lmax, with 4, 2 and 1 times the maps."""
    parts = []
    for div, times in ((4, 4), (2, 2), (1, 1)):
        lmax = max(8, c["lmax"] // div)
        nphi = 16
        while nphi < 2 * lmax + 2:
            nphi *= 2
        nrings = max(lmax + 1, c["nrings"] // div) if div > 1 else c["nrings"]
        parts.append(dict(c, kind="beta", lmax=lmax, nrings=nrings, nphi=nphi, maps=c["maps"] * times))
    return parts


def _cov_sims(n):
    return 2 * n + 16


def _plan(c):
    ring_mask, pix_mask = _mask(c)
    plan = M.Plan(c["lmax"], c["P"], _basis(c["lmax"], c["P"]), _cl(c["lmax"]), c["nrings"], c["nphi"],
                  prec=c["prec"], ring_mask=ring_mask, pix_mask=pix_mask)
    if c["lmax"] >= 2000:
        plan.set_chunk(c["maps"])
    if c["linear"] == "ring":
        plan.set_linear_mode("ring")
    return plan


def _means(plan, c, seed, stream=1):
    if c["sims"] > 0:
        plan.linear_term(_alm(c["lmax"], c["sims"], seed, stream), finalize=True)


def prepare(case, seed):
    c = dict(case)
    kind = c["kind"]
    if kind == "batch":
        parts = _batch_parts(c)
        plans = [_plan(p) for p in parts]
        for i, (plan, p) in enumerate(zip(plans, parts)):
            _means(plan, p, seed, 1 + 2 * i)
        alms = [_alm(p["lmax"], p["maps"], seed, 2 + 2 * i) for i, p in enumerate(parts)]
        return {"kind": kind, "batch": M.Batch(plans), "alms": alms, "linear": c["linear"] != "none"}
    plan = _plan(c)
    st = {"kind": kind, "plan": plan, "linear": c["linear"] != "none"}
    if kind != "means":
        _means(plan, c, seed)
    if kind == "alm":
        st["noise"] = torch.randn((c["maps"], c["nrings"], c["nphi"]), generator=_gen(seed, 3), device="cuda")
    elif kind == "solve":
        st["beta"] = _betas(plan.n_max, c["maps"], seed, 4)
        st["alpha"] = _alpha(plan.n_max, seed)
        plan.cov_accumulate(_betas(plan.n_max, _cov_sims(plan.n_max), seed, 5))
    else:
        st["alm"] = _alm(c["lmax"], c["maps"], seed, 2)
    if kind == "grad":
        st["g"] = torch.randn((c["maps"], plan.n_max), generator=_gen(seed, 6), device="cuda", dtype=torch.float64)
    if kind == "fnl":
        st["alpha"] = _alpha(plan.n_max, seed)
        st["grad_out"] = torch.randn(c["maps"], generator=_gen(seed, 7), device="cuda", dtype=torch.float64)
        plan.cov_accumulate(_betas(plan.n_max, _cov_sims(plan.n_max), seed, 5))
    return st


def run(s):
    kind = s["kind"]
    if kind == "batch":
        return list(s["batch"].cubic(s["alms"], use_linear=s["linear"]))
    plan = s["plan"]
    if kind == "beta":
        return plan.cubic(s["alm"], use_linear=s["linear"])
    if kind == "means":
        plan.reset(1)                                  # a new estimate of the means
        plan.linear_term(s["alm"], finalize=True)
        return plan.pair_mean()
    if kind == "grad":
        return plan.backward(s["alm"], s["g"], use_linear=s["linear"])
    if kind == "maps":
        return plan.synthesize(s["alm"])
    if kind == "alm":
        return plan.analyze(s["noise"])
    if kind == "tau":
        return plan.quartic(s["alm"], use_linear=s["linear"])
    if kind == "solve":
        fnl, sigma = plan.solve(s["alpha"], s["beta"])
        w, _ = plan.fnl_weights(s["alpha"])
        return {"fnl": fnl, "sigma": sigma, "w": w}
    if kind == "fnl":
        a = s["alm"].detach().requires_grad_(True)
        fnl = M.modal_fnl(a, plan, s["alpha"], use_linear=s["linear"])
        (grad,) = torch.autograd.grad(fnl, a, s["grad_out"])
        return {"fnl": fnl.detach(), "grad": grad}
    raise ValueError("unknown kind %r" % kind)


def work(case):
    """Bytes: a_lm or maps in, results out (pair means in where they are used per pixel); flops: the separable
    algorithm's sums (Legendre, FFT, products), a multiply-add as 2."""
    c = dict(case)
    kind, P, B, R, N, L = c["kind"], c["P"], c["maps"], c["nrings"], c["nphi"], c["lmax"]
    if kind == "batch":
        parts = [work(p) for p in _batch_parts(c)]
        return {k: sum(p[k] for p in parts) for k in ("bytes", "flops")}
    npix, n_alm, n_max, n_pair = R * N, _n_alm(L), _n_modes(P), P * (P + 1) // 2
    if kind == "solve":
        n = n_max
        return {"bytes": 8.0 * (n * n + (B + 2) * n), "flops": n ** 3 / 3.0 + 2.0 * n * n + (B + 2.0) * n * n}
    leg = 4.0 * n_alm * ((R + 1) // 2) * B               # one channel of B maps, one direction
    fft = 2.5 * npix * math.log2(N) * B
    alm, synth = 8.0 * n_alm * B, P * (leg + fft)
    if kind == "alm":
        return {"bytes": alm + 4.0 * npix * B, "flops": leg + fft}
    if kind == "maps":
        return {"bytes": alm + 4.0 * npix * P * B, "flops": synth}
    if kind == "means":
        return {"bytes": alm + 4.0 * n_pair * npix, "flops": synth + 2.0 * n_pair * npix * B}
    means = {"none": 0.0, "pixel": 4.0 * n_pair * npix, "ring": 8.0 * n_pair * R}[c["linear"]]
    lin = {"none": 0.0, "pixel": 2.0 * n_pair * P * npix * B, "ring": 2.0 * n_pair * P * R * B}[c["linear"]]
    cubic = 2.0 * n_max * npix * B
    if kind == "beta":
        return {"bytes": alm + means + 8.0 * n_max * B, "flops": synth + cubic + lin}
    if kind == "tau":
        n_quad = n_max * (P + 3) // 4
        return {"bytes": alm + means + 8.0 * n_quad * B, "flops": synth + 2.0 * n_quad * npix * B}
    back = {"bytes": 2.0 * alm + means + 8.0 * n_max * B, "flops": 2.0 * synth + 3.0 * cubic + lin}
    if kind == "grad":
        return back
    return {"bytes": back["bytes"] + 8.0 * n_max * n_max,
            "flops": back["flops"] + cubic + lin + n_max ** 3 / 3.0 + (B + 2.0) * n_max * n_max}


# ------------------------------------------------------------------ the same in 64 bits, plain torch

def _gl(n):
    x, w = np.polynomial.legendre.leggauss(n) if n < 200 else _gl_newton(n)
    return x[::-1].copy(), w[::-1].copy()                 # north first


def _gl_newton(n):
    k = np.arange(n, dtype=float)
    x = -np.cos(np.pi * (k + 0.75) / (n + 0.5))
    for _ in range(8):
        p0, p1 = np.ones_like(x), x.copy()
        for i in range(2, n + 1):
            p0, p1 = p1, ((2 * i - 1) * x * p1 - (i - 1) * p0) / i
        dp = n * (x * p1 - p0) / (x * x - 1.0)
        x = x - p1 / dp
    x = 0.5 * (x - x[::-1])
    p0, p1 = np.ones_like(x), x.copy()
    for i in range(2, n + 1):
        p0, p1 = p1, ((2 * i - 1) * x * p1 - (i - 1) * p0) / i
    dp = n * (x * p1 - p0) / (x * x - 1.0)
    return x, 2.0 / ((1.0 - x * x) * dp * dp)


class _Sphere:
    """Legendre functions of the northern half of the rings and the transforms of one grid, float64."""

    def __init__(self, lmax, nrings, nphi):
        self.L, self.R, self.N, self.H = lmax, nrings, nphi, (nrings + 1) // 2
        mu, w = _gl(nrings)
        self.w = torch.from_numpy(w).cuda()
        x = torch.from_numpy(mu[:self.H]).cuda()
        L1 = lmax + 1
        m = torch.arange(L1, device="cuda", dtype=torch.float64)
        k = torch.arange(1, L1, device="cuda", dtype=torch.float64)
        lp = torch.cat([torch.zeros(1, device="cuda", dtype=torch.float64), torch.cumsum(torch.log2((2 * k - 1) / (2 * k)), 0)])
        l2 = 0.5 * (torch.log2((2 * m + 1) / (4 * math.pi)) + lp)[:, None] + 0.5 * m[:, None] * torch.log2(1 - x * x)[None, :]
        e = torch.floor(l2)
        sign = torch.where(torch.arange(L1, device="cuda") % 2 == 1, -1.0, 1.0).double()
        v = sign[:, None] * torch.exp2(l2 - e)            # lambda = v 2^e
        self.lam = torch.zeros((L1, L1, self.H), device="cuda", dtype=torch.float64)       # [d = l - m][m][ring]
        prev = torch.zeros_like(v)
        for d in range(L1):
            n = L1 - d
            if d > 0:
                mm = m[:n]
                l = mm + d
                a = torch.sqrt((4 * l * l - 1) / (l * l - mm * mm))
                b = torch.sqrt(((l - 1) ** 2 - mm * mm).clamp(min=0) / (4 * (l - 1) ** 2 - 1))
                v, prev, e = a[:, None] * (x[None, :] * v[:n] - b[:, None] * prev[:n]), v[:n], e[:n]
                if d % 8 == 0:
                    big = v.abs() > 2.0 ** 100
                    s = torch.where(big, 2.0 ** -100, 1.0).double()
                    v, prev, e = v * s, prev * s, e + 100.0 * big
            half = torch.exp2((0.5 * e).floor().clamp(min=-1000))
            self.lam[d, :n] = v * half * torch.exp2((e - (0.5 * e).floor()).clamp(min=-1000))

    def _start(self, m):
        return m * (2 * self.L + 3 - m) // 2

    def maps(self, fa):
        """fa complex128 [C][n_alm] -> maps [C][R][N]."""
        C, S = fa.shape[0], self.R // 2
        D = torch.zeros((C, self.R, self.N // 2 + 1), device="cuda", dtype=torch.complex128)
        for m in range(self.L + 1):
            i, n = self._start(m), self.L + 1 - m
            a = torch.view_as_real(fa[:, i:i + n])
            z = [torch.einsum("cdr,dj->cjr", a[:, p::2], self.lam[p:n:2, m]) if n > p else 0.0 for p in (0, 1)]
            D[:, :self.H, m] = torch.view_as_complex((z[0] + z[1]).contiguous())
            south = torch.view_as_complex((z[0] - z[1]).contiguous())[:, :S]
            D[:, self.R - S:, m] = south.flip(1)
        D[..., 0] = D[..., 0].real.to(torch.complex128)
        return torch.fft.irfft(D, n=self.N, dim=2, norm="forward")

    def adjoint(self, u):
        """u [C][R][N] -> complex128 [C][n_alm]: sum_x u(x) lambda_lm e^{-i m phi}."""
        C, S = u.shape[0], self.R // 2
        F = torch.fft.rfft(u, dim=2)[..., :self.L + 1]
        north = F[:, :self.H]
        south = torch.zeros_like(north)
        south[:, :S] = F[:, self.R - S:].flip(1)
        out = torch.zeros((C, _n_alm(self.L)), device="cuda", dtype=torch.complex128)
        for m in range(self.L + 1):
            i, n = self._start(m), self.L + 1 - m
            for p, z in ((0, north[..., m] + south[..., m]), (1, north[..., m] - south[..., m])):
                if n > p:
                    g = torch.einsum("dj,cjr->cdr", self.lam[p:n:2, m], torch.view_as_real(z.contiguous()))
                    out[:, i + p:i + n:2] = torch.view_as_complex(g.contiguous())
        return out


class _Exact:
    """One plan's path in float64."""

    def __init__(self, c):
        self.c, self.P, self.L = c, c["P"], c["lmax"]
        self.sphere = _Sphere(c["lmax"], c["nrings"], c["nphi"])
        cl = _cl(self.L)
        f = np.where(cl > 0, _basis(self.L, self.P) / np.sqrt(np.where(cl > 0, cl, 1.0)), 0.0)
        self.l, self.m = _lm(self.L)
        self.f = torch.from_numpy(f).cuda()[:, self.l]   # [P][n_alm]
        W = (self.sphere.w * (TWO_PI / c["nphi"]))[:, None].repeat(1, c["nphi"])
        ring_mask, pix_mask = _mask(c)
        if ring_mask is not None:
            W = W * torch.from_numpy(ring_mask).cuda().double()[:, None]
        if pix_mask is not None:
            W = W * torch.from_numpy(pix_mask).cuda().double()
        self.W = W.reshape(-1)
        self.pairs = [(a, b) for a in range(self.P) for b in range(a, self.P)]
        self.pa = torch.tensor([a for a, _ in self.pairs], device="cuda")
        self.pb = torch.tensor([b for _, b in self.pairs], device="cuda")
        num = np.zeros((self.P, self.P), dtype=np.int64)
        for i, (a, b) in enumerate(self.pairs):
            num[a, b] = num[b, a] = i
        self.num = torch.from_numpy(num).cuda()
        self.mean = None

    def synth(self, alm):
        """alm complex64 [n_alm] -> [P][npix]."""
        return self.sphere.maps(self.f * alm.to(torch.complex128)).reshape(self.P, -1)

    def set_means(self, seed, stream=1):
        if self.c["sims"] > 0:
            sims = _alm(self.L, self.c["sims"], seed, stream)
            self.mean = self.pair_mean(sims)

    def pair_mean(self, sims):
        s = 0.0
        for i in range(sims.shape[0]):
            X = self.synth(sims[i])
            s = s + X[self.pa] * X[self.pb]
        s = s / sims.shape[0]
        if self.c["linear"] == "ring":
            R, N = self.c["nrings"], self.c["nphi"]
            s = s.reshape(-1, R, N).mean(2, keepdim=True).expand(-1, R, N).reshape(len(self.pairs), -1)
        return s

    def triples(self):
        P = self.P
        t = [(p, r, s) for p in range(P) for r in range(p, P) for s in range(r, P)]
        return torch.tensor(t, device="cuda").T

    def beta(self, X):
        p, r, s = self.triples()
        C = torch.zeros((len(self.pairs), self.P), device="cuda", dtype=torch.float64)
        G = torch.zeros_like(C)
        for x in range(0, X.shape[1], 1 << 20):
            V = X[:, x:x + (1 << 20)]
            C += (V[self.pa] * V[self.pb] * self.W[x:x + (1 << 20)]) @ V.T
            if self.mean is not None:
                G += (self.mean[:, x:x + (1 << 20)] * self.W[x:x + (1 << 20)]) @ V.T
        n = self.num
        return C[n[p, r], s] - (G[n[p, r], s] + G[n[p, s], r] + G[n[r, s], p])

    def tau(self, X):
        P = self.P
        q = torch.tensor([(a, b, c, d) for a in range(P) for b in range(a, P) for c in range(b, P) for d in range(c, P)],
                         device="cuda").T
        Q = X[self.pa] * X[self.pb]
        T = (Q * self.W) @ Q.T
        n = self.num
        out = T[n[q[0], q[1]], n[q[2], q[3]]].clone()
        if self.mean is not None:
            H = (self.mean * self.W) @ Q.T
            K = (self.mean * self.W) @ self.mean.T
            for i, j, k, o in ((0, 1, 2, 3), (0, 2, 1, 3), (0, 3, 1, 2), (1, 2, 0, 3), (1, 3, 0, 2), (2, 3, 0, 1)):
                out -= H[n[q[i], q[j]], n[q[k], q[o]]]
            for i, j, k, o in ((0, 1, 2, 3), (0, 2, 1, 3), (0, 3, 1, 2)):
                out += K[n[q[i], q[j]], n[q[k], q[o]]]
        return out

    def grad(self, X, g):
        """Gradient of sum_n g_n beta_n with respect to (Re a_lm, Im a_lm), complex128 [n_alm]."""
        p, r, s = self.triples()
        h = torch.zeros((self.P,) * 3, device="cuda", dtype=torch.float64)
        perms = ((p, r, s), (p, s, r), (r, p, s), (r, s, p), (s, p, r), (s, r, p))
        distinct = torch.where((p == r) & (r == s), 1.0, torch.where((p == r) | (r == s), 3.0, 6.0)).double()
        for i, j, k in perms:
            h[i, j, k] = g / distinct
        hk = h[:, self.pa, self.pb] * torch.where(self.pa == self.pb, 1.0, 2.0).double()
        U = torch.empty_like(X)
        for x in range(0, X.shape[1], 1 << 20):
            V = X[:, x:x + (1 << 20)]
            Q = V[self.pa] * V[self.pb]
            if self.mean is not None:
                Q = Q - self.mean[:, x:x + (1 << 20)]
            U[:, x:x + (1 << 20)] = 3.0 * self.W[x:x + (1 << 20)] * (hk @ Q)
        a = self.sphere.adjoint(U.reshape(self.P, self.c["nrings"], self.c["nphi"]))
        out = (self.f * a).sum(0) * torch.where(self.m == 0, 1.0, 2.0).double()
        return torch.where(self.m == 0, out.real.to(torch.complex128), out)


def _exact_solve(n, seed, alpha, beta):
    sims = _betas(n, _cov_sims(n), seed, 5)
    zeta = torch.cov(sims.T) / 6.0
    a = torch.from_numpy(alpha).cuda()
    x = torch.linalg.solve(zeta, a)
    norm = a @ x
    return beta @ x / norm, math.sqrt(6.0 / float(norm)), x / norm


def exact(case, seed):
    c = dict(case)
    kind = c["kind"]
    if kind == "batch":
        out = []
        for i, p in enumerate(_batch_parts(c)):
            e = _Exact(p)
            e.set_means(seed, 1 + 2 * i)
            alm = _alm(p["lmax"], p["maps"], seed, 2 + 2 * i)
            out.append(torch.stack([e.beta(e.synth(a)) for a in alm]))
        return out
    n = _n_modes(c["P"])
    if kind == "solve":
        fnl, sigma, w = _exact_solve(n, seed, _alpha(n, seed), _betas(n, c["maps"], seed, 4))
        return {"fnl": fnl.cpu().numpy(), "sigma": sigma, "w": w}
    if kind == "alm":
        sph = _Sphere(c["lmax"], c["nrings"], c["nphi"])
        noise = torch.randn((c["maps"], c["nrings"], c["nphi"]), generator=_gen(seed, 3), device="cuda")
        return sph.adjoint(noise.double() * (sph.w * (TWO_PI / c["nphi"]))[None, :, None])
    e = _Exact(c)
    alm = _alm(c["lmax"], c["maps"], seed, 2)
    if kind == "means":
        return e.pair_mean(alm)
    if kind == "maps":
        return torch.stack([e.synth(a).reshape(c["P"], c["nrings"], c["nphi"]) for a in alm])
    e.set_means(seed)
    if kind == "beta":
        return torch.stack([e.beta(e.synth(a)) for a in alm])
    if kind == "tau":
        return torch.stack([e.tau(e.synth(a)) for a in alm])
    if kind == "grad":
        g = torch.randn((c["maps"], n), generator=_gen(seed, 6), device="cuda", dtype=torch.float64)
        return torch.stack([e.grad(e.synth(a), g[b]) for b, a in enumerate(alm)])
    beta = torch.stack([e.beta(e.synth(a)) for a in alm])
    fnl, _, w = _exact_solve(n, seed, _alpha(n, seed), beta)
    go = torch.randn(c["maps"], generator=_gen(seed, 7), device="cuda", dtype=torch.float64)
    return {"fnl": fnl, "grad": torch.stack([e.grad(e.synth(a), go[b] * w) for b, a in enumerate(alm)])}
