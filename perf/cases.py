"""The transforms whose speed is measured, their inputs, and their exact results.

A case is one use of the library through ``paper_2406_14542_gb300``: a kind of
call (``synth``, ``adjoint``, ``step`` = both, ``autograd``, ``spin``,
``pointing``, ``batch``) on one band limit and point set.  ``exact`` evaluates
the same transforms in 64 bits with plain torch: the textbook normalised
Legendre (or Wigner-d) recurrence on rings, torch's FFTs, and Kaiser-Bessel
gridding of width 16 on a twofold grid (truncation below 1e-14).
"""
import math
import random

import numpy as np
import torch

import paper_2406_14542_gb300 as nu

ARCMIN = math.pi / (180.0 * 60.0)


def listed():
    return [
        # the smallest call: a low-resolution map at scattered points, where
        # launches and the serial recurrence are the time
        dict(name="fp64_63_synth", kind="synth", precision="fp64", eps=1e-10, lmax=63, points="sphere", npts=20000),
        dict(name="fp64_63_adjoint", kind="adjoint", precision="fp64", eps=1e-10, lmax=63, points="sphere", npts=20000),
        # an odd band limit with fewer orders than degrees on a survey
        # footprint: points crowded in one patch, an odd number of them
        dict(name="fp64_517_patch_step", kind="step", precision="fp64", eps=1e-8, lmax=517, mmax=301, points="patch",
             npts=123457),
        # lensed CMB maps at three resolutions: a Gauss-Legendre ring grid
        # deflected by 2.5 arcmin; one iteration of a map solver is a
        # synthesis and an adjoint
        dict(name="fp64_1023_step", kind="step", precision="fp64", eps=1e-10, lmax=1023, points="rings"),
        dict(name="mixed_2047_step", kind="step", precision="mixed", eps=1e-5, lmax=2047, points="rings"),
        dict(name="fp64_4095_synth", kind="synth", precision="fp64", eps=1e-10, lmax=4095, points="rings"),
        dict(name="fp64_4095_adjoint", kind="adjoint", precision="fp64", eps=1e-10, lmax=4095, points="rings"),
        # a differentiable loss: forward, and the gradients in a_lm and in the
        # point coordinates
        dict(name="fp64_2047_autograd", kind="autograd", precision="fp64", eps=1e-10, lmax=2047, points="rings"),
        # polarisation: spin 2, both directions
        dict(name="spin2_1023_step", kind="spin", precision="fp64", eps=1e-10, lmax=1023, spin=2, points="rings"),
        # the deflected coordinates of a ring grid from a lensing potential
        dict(name="pointing_2047", kind="pointing", precision="fp64", eps=1e-10, lmax=2047, points="grid"),
        # many transforms of uneven band limit (a simulation suite), 2 lmax^2
        # scattered points each, both directions
        dict(name="batch32_mixed_step", kind="batch", precision="mixed", eps=1e-5, lmin=256, lmax=1535, members=32),
        dict(name="batch16_fp64_step", kind="batch", precision="fp64", eps=1e-10, lmin=256, lmax=1023, members=16),
    ]


def draw(rng: random.Random):
    kind = rng.choice(["synth", "adjoint", "step", "step", "autograd", "spin", "pointing", "batch"])
    precision = "fp64" if kind in ("spin", "pointing") else rng.choice(["fp64", "fp64", "mixed"])
    eps = rng.choice([1e-6, 1e-8, 1e-10, 1e-10, 1e-12] if precision == "fp64" else [1e-3, 1e-4, 1e-5, 1e-5])

    def log_int(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    c = dict(kind=kind, precision=precision, eps=eps)
    if kind == "batch":
        lmax = log_int(100, 1023)
        c.update(lmin=max(16, int(lmax * rng.uniform(0.1, 0.8))), lmax=lmax, members=rng.randint(3, 16))
        return c
    c["lmax"] = log_int(40, 1023 if kind == "spin" else 2047)
    c["points"] = "grid" if kind == "pointing" else rng.choice(["rings", "sphere", "patch"])
    if c["points"] in ("sphere", "patch"):
        c["npts"] = log_int(2000, min(8000000, 4 * (c["lmax"] + 1) ** 2))
    if kind == "spin":
        c["spin"] = rng.choice([1, 2, 2, 3])
    elif kind in ("synth", "adjoint", "step") and rng.random() < 0.25:
        c["mmax"] = int(c["lmax"] * rng.uniform(0.3, 0.95))
    if kind in ("adjoint", "step") and precision == "fp64" and rng.random() < 0.2:
        c["deterministic"] = True
    return c


# ---------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------
def _gen(seed, k):
    g = torch.Generator(device="cuda")
    g.manual_seed((int(seed) * 1000003 + k) % (1 << 62))
    return g


def _rand(n, g):
    return torch.rand(n, generator=g, device="cuda", dtype=torch.float64)


def _randn(n, g):
    return torch.randn(n, generator=g, device="cuda", dtype=torch.float64)


def _ells(lmax, mmax):
    return torch.from_numpy(np.concatenate([np.arange(m, lmax + 1) for m in range(mmax + 1)])).cuda()


def _alm(lmax, mmax, g):
    """Gaussian coefficients with C_l = (l + 1)^-2, m-major; the m = 0 block real."""
    n = nu.nalm(lmax, mmax)
    a = torch.complex(_randn(n, g), _randn(n, g)) * math.sqrt(0.5)
    a[: lmax + 1] = a[: lmax + 1].real * math.sqrt(2.0) + 0j
    return a / (_ells(lmax, mmax) + 1.0)


def _phi_lm(lmax, g, rms=2.5 * ARCMIN):
    """Lensing-like potential: C_l ~ [l(l+1)]^-1 (1 + l/60)^-3 for l >= 2, scaled to the rms deflection."""
    l = torch.arange(lmax + 1, dtype=torch.float64, device="cuda")
    cl = torch.where(l >= 2, 1.0 / (l * (l + 1)).clamp(min=1) / (1 + l / 60) ** 3, torch.zeros_like(l))
    cl = cl * rms**2 / ((2 * l + 1) * l * (l + 1) * cl).sum() * 4 * math.pi
    a = _alm(lmax, lmax, g)
    e = _ells(lmax, lmax)
    return a * (e + 1.0) * cl.sqrt()[e]


def _rings(lmax, nphi, phi0=0.0):
    """(lmax + 1) x nphi ring grid at the Gauss-Legendre colatitudes (to O(n^-4)), phi from phi0 pixels on."""
    n = lmax + 1
    k = torch.arange(1, n + 1, dtype=torch.float64, device="cuda")
    x = (1 - 1 / (8.0 * n * n) + 1 / (8.0 * n**3)) * torch.cos(math.pi * (4 * k - 1) / (4 * n + 2))
    ph = 2 * math.pi / nphi * (torch.arange(nphi, dtype=torch.float64, device="cuda") + phi0)
    return torch.stack([torch.acos(x).repeat_interleave(nphi), ph.repeat(n)], dim=1)


def _shift(th, ph, at, ap):
    """Each point moved along the great circle in direction (at, ap) by |(at, ap)|."""
    al = torch.sqrt(at * at + ap * ap)
    sc = torch.where(al > 0, torch.sin(al) / al.clamp(min=1e-300), torch.ones_like(al))
    ca, st, ct, sp, cp = torch.cos(al), torch.sin(th), torch.cos(th), torch.sin(ph), torch.cos(ph)
    x = ca * st * cp + sc * (at * ct * cp - ap * sp)
    y = ca * st * sp + sc * (at * ct * sp + ap * cp)
    z = ca * ct - sc * at * st
    return torch.stack([torch.atan2(torch.sqrt(x * x + y * y), z), torch.remainder(torch.atan2(y, x), 2 * math.pi)], 1)


def _deflected(lmax, g, rms=2.5 * ARCMIN):
    """The (lmax + 1) x (2 lmax + 1) ring grid moved by the gradient of a random smooth potential (16 plane waves), in ring order."""
    pts = _rings(lmax, 2 * lmax + 1)
    q = torch.randn((16, 3), generator=g, device="cuda", dtype=torch.float64)
    q = q / q.norm(dim=1, keepdim=True) * (20 + 60 * _rand(16, g))[:, None]
    d = 2 * math.pi * _rand(16, g)
    amp = rms / math.sqrt(16 / 3.0) / q.norm(dim=1)
    out = torch.empty_like(pts)
    for i in range(0, pts.shape[0], 1 << 22):
        th, ph = pts[i : i + (1 << 22)].unbind(1)
        st, ct, sp, cp = torch.sin(th), torch.cos(th), torch.sin(ph), torch.cos(ph)
        at, ap = torch.zeros_like(th), torch.zeros_like(th)
        for k in range(16):
            qx, qy, qz = (float(v) for v in q[k])
            t = -float(amp[k]) * torch.sin(st * (qx * cp + qy * sp) + qz * ct + float(d[k]))
            at += t * (ct * (qx * cp + qy * sp) - qz * st)
            ap += t * (qy * cp - qx * sp)
        out[i : i + (1 << 22)] = _shift(th, ph, at, ap)
    return out


def _points(case, g):
    lmax = case["lmax"]
    if case["points"] == "grid":  # pixel centres half a pixel off the meridian
        return _rings(lmax, 2 * lmax + 2, 0.5)
    if case["points"] == "rings":
        return _deflected(lmax, g)
    n = case["npts"]
    if case["points"] == "sphere":
        return torch.stack([torch.acos(2 * _rand(n, g) - 1), 2 * math.pi * _rand(n, g)], dim=1)
    # a footprint of about 30 by 60 degrees, denser towards its middle
    th = 0.9 + 0.25 * (_rand(n, g) + _rand(n, g) - 1)
    ph = 2.0 + 0.5 * (_rand(n, g) + _rand(n, g) - 1)
    return torch.stack([th, ph], dim=1)


def _mmax(case):
    return case.get("mmax") or case["lmax"]


def _inputs(case, seed):
    """Everything in 64 bits; prepare() rounds to the case's types."""
    fp = (lambda t: t) if case["precision"] == "fp64" else (lambda t: t.to(torch.complex64 if t.is_complex() else torch.float32))
    if case["kind"] == "batch":
        r = random.Random(case["lmax"] * 977 + case["members"])  # the suite's band limits; its data come from the seed
        out = []
        for b in range(case["members"]):
            l = case["lmax"] if b == 0 else r.randint(case["lmin"], case["lmax"])
            g = _gen(seed, 17 + b)
            p = _points(dict(lmax=l, points="sphere", npts=2 * l * l), g)
            out.append((l, p, fp(_alm(l, l, g)), fp(_randn(p.shape[0], g))))
        return out
    g = _gen(seed, 1)
    pts = _points(case, g)
    n, L, mm = pts.shape[0], case["lmax"], _mmax(case)
    k = case["kind"]
    if k == "pointing":
        return dict(pts=pts, phi=fp(_phi_lm(L, g)))
    s = dict(pts=pts)
    if k in ("synth", "step", "autograd", "spin"):
        s["a"] = fp(_alm(L, mm, g))
    if k in ("adjoint", "step", "spin"):
        s["y"] = fp(_randn(n, g))
    if k == "spin":
        s["c"], s["u"] = _alm(L, mm, g), _randn(n, g)
        e = _ells(L, mm)
        s["a"][e < case["spin"]] = 0
        s["c"][e < case["spin"]] = 0
    if k == "autograd":
        s["w"] = fp(_rand(n, g))
    return s


def prepare(case, seed):
    if case["kind"] == "batch":
        m = _inputs(case, seed)
        plan = nu.BatchPlan([x[0] for x in m], [x[1] for x in m], eps=case["eps"], precision=case["precision"])
        return dict(kind="batch", plan=plan, a=[x[2] for x in m], y=[x[3] for x in m])
    s = _inputs(case, seed)
    s["kind"] = case["kind"]
    s["plan"] = nu.Plan(case["lmax"], s["pts"], eps=case["eps"], precision=case["precision"], mmax=case.get("mmax"),
                        spin=case.get("spin", 0), deterministic=bool(case.get("deterministic")))
    if case["kind"] == "autograd":
        s["a"].requires_grad_()
        s["pts"].requires_grad_()
    return s


def run(state):
    plan, k = state["plan"], state["kind"]
    if k == "synth":
        return plan.synth(state["a"])
    if k == "adjoint":
        return plan.adjoint(state["y"])
    if k in ("step", "batch"):
        return dict(map=plan.synth(state["a"]), alm=plan.adjoint(state["y"]))
    if k == "spin":
        q, u = plan.synth_spin(state["a"], state["c"])
        g, c = plan.adjoint_spin(state["y"], state["u"])
        return dict(q=q, u=u, g=g, c=c)
    if k == "pointing":
        return plan.pointing(state["phi"])
    f = nu.nusht(state["a"], state["pts"], plan)
    loss = (state["w"] * f * f).sum()
    ga, gp = torch.autograd.grad(loss, (state["a"], state["pts"]))
    return dict(map=f.detach(), grad_alm=ga, grad_pts=gp)


# ---------------------------------------------------------------------------
# work
# ---------------------------------------------------------------------------
def _one_way(L, mm, n, eps, spin=0):
    """Operations of one direction: per (ring pair, l, m) one recurrence
    multiply-add and one complex multiply-add (twice both for spin), the two
    2D half-size FFTs, and w^2 taps a point."""
    pairs, nalm = (L + 2) // 2, nu.nalm(L, mm)
    w = math.ceil(-math.log10(eps)) + 2
    grid = (3 * L + 2) ** 2
    one = 2.5 * grid * math.log2(grid) + 2.0 * n * w * w
    return pairs * nalm * 6.0 * (4 if spin else 1) + one * (2 if spin else 1)


def work(case):
    r = 8 if case["precision"] == "fp64" else 4
    if case["kind"] == "batch":
        rnd = random.Random(case["lmax"] * 977 + case["members"])
        by = fl = 0.0
        for b in range(case["members"]):
            l = case["lmax"] if b == 0 else rnd.randint(case["lmin"], case["lmax"])
            by += 2 * (2 * l * l * (16 + r) + nu.nalm(l) * 2 * r)
            fl += 2 * _one_way(l, l, 2 * l * l, case["eps"])
        return dict(bytes=by, flops=fl)
    L, mm, k = case["lmax"], _mmax(case), case["kind"]
    n = case.get("npts") or (L + 1) * (2 * L + (2 if case["points"] == "grid" else 1))
    fl = _one_way(L, mm, n, case["eps"], case.get("spin", 0))
    a = nu.nalm(L, mm) * 2 * r
    if k == "pointing":
        return dict(bytes=a + n * 32.0, flops=fl)
    if k == "spin":
        return dict(bytes=2.0 * (n * (16 + 2 * r) + 2 * a), flops=2 * fl)
    if k == "autograd":  # map, cotangent and weights; gradients in a_lm and in the points
        return dict(bytes=2.0 * a + n * (32.0 + 3 * r), flops=3 * fl)
    ways = 2 if k == "step" else 1
    return dict(bytes=float(ways * (n * (16 + r) + a)), flops=ways * fl)


# ---------------------------------------------------------------------------
# the same transforms in 64 bits, plain torch
# ---------------------------------------------------------------------------
_STEP, _TINY = 900, -600  # values below 2^-600 are carried as p 2^(-900 k)


def _power(s, e):
    """s^e as (mantissa, binary exponent): s^(e/8) is formed by pow, then raised to the eighth."""
    t, x = torch.frexp(torch.pow(s, e / 8.0))
    dead = t == 0
    t = torch.where(dead, torch.ones_like(t), t)
    return t**8, torch.where(dead, torch.full_like(x, -60000), 8 * x).to(torch.int64)


class _Chain:
    """Rows m = 0..mmax of a three-term recurrence on the rings, a row started at its first degree."""

    def __init__(self, mant, expo):
        k = torch.clamp((_TINY - expo + _STEP - 1) // _STEP, min=0)
        self.k = k.to(torch.int32)
        self.p = torch.ldexp(mant, (expo + _STEP * k).clamp(-1000, 1000).to(torch.int32))
        self.q = torch.zeros_like(self.p)

    def step(self, rows, fa, fb, x, fc):
        """p <- (fa x + fb) p - fc q on the first `rows` rows."""
        t = fa[:rows, None] * x
        if fb is not None:
            t += fb[:rows, None]
        t *= self.p[:rows]
        t -= fc[:rows, None] * self.q[:rows]
        self.q[:rows] = self.p[:rows]
        self.p[:rows] = t

    def settle(self):
        up = (self.p.abs() > 2.0**300) & (self.k > 0)
        f = torch.where(up, torch.full_like(self.p, 2.0**-_STEP), torch.ones_like(self.p))
        self.p *= f
        self.q *= f
        self.k -= up.to(torch.int32)
        self.live = (self.k == 0).to(self.p.dtype)

    def value(self, rows):
        return self.p[:rows] * self.live[:rows]


def _good(n):
    while True:
        r = n
        for f in (2, 3, 5):
            while r % f == 0:
                r //= f
        if r == 1 and n % 4 == 0:
            return n
        n += 1


def _legendre(L, mm, M):
    """Yields (l, rows, P): the normalised P_l^m at theta_j = 2 pi j / M, j = 0..M/2, for m < rows."""
    th = 2 * math.pi / M * torch.arange(M // 2 + 1, dtype=torch.float64, device="cuda")
    x, s = torch.cos(th), torch.sin(th).clamp(min=0)
    s[-1] = 0
    m = torch.arange(mm + 1, dtype=torch.float64, device="cuda")
    c = torch.sqrt(torch.cumprod(torch.where(m > 0, (2 * m + 1) / (2 * m).clamp(min=1), 1 / (4 * math.pi)), 0))
    c = torch.where(m % 2 == 1, -c, c)
    mant, ex = _power(s[None, :], m[:, None])
    ch = _Chain(c[:, None] * mant, ex)
    ch.settle()
    al = lambda l: torch.sqrt(((l * l - m * m) / (4.0 * l * l - 1)).clamp(min=0))  # noqa: E731
    for l in range(L + 1):
        rows = min(l, mm + 1)  # orders below l advance, order l starts
        if rows:
            a1 = al(l)
            ch.step(rows, 1 / a1, None, x, al(l - 1) / a1)
        if l % 16 == 0:
            ch.settle()
        rows = min(l + 1, mm + 1)
        yield l, rows, ch.value(rows)


def _wigner(L, M, spin):
    """Yields (l, rows, lambda+, lambda-): spin +-s functions at phi = 0, as _legendre."""
    th = 2 * math.pi / M * torch.arange(M // 2 + 1, dtype=torch.float64, device="cuda")
    x, c, s = torch.cos(th), torch.cos(th / 2), torch.sin(th / 2)
    c[-1] = 0
    m = torch.arange(L + 1, dtype=torch.float64, device="cuda")
    chains = []
    for sp in (-spin, spin):
        mant, expo, pa, pb = [], [], [], []
        for k in range(L + 1):
            l0 = max(k, spin)
            if k >= spin:
                a, b, binom, neg = l0 + sp, l0 - sp, math.comb(2 * l0, l0 + sp), (l0 - sp) & 1
            elif sp > 0:
                a, b, binom, neg = l0 + k, l0 - k, math.comb(2 * l0, l0 + k), 0
            else:
                a, b, binom, neg = l0 - k, l0 + k, math.comb(2 * l0, l0 - k), (l0 + k) & 1
            e = binom.bit_length() // 2 * 2
            v = math.sqrt(binom / 2**e) * math.sqrt((2 * l0 + 1) / (4 * math.pi))
            mant.append(-v if (neg + spin) & 1 else v)
            expo.append(e // 2)
            pa.append(a)
            pb.append(b)
        t = lambda v: torch.tensor(v, dtype=torch.float64, device="cuda")[:, None]  # noqa: E731
        (ma, ea), (mb, eb) = _power(c[None, :], t(pa)), _power(s[None, :], t(pb))
        chains.append(_Chain(t(mant) * ma * mb, ea + eb + t(expo).to(torch.int64)))
        chains[-1].settle()
    for l in range(spin, L + 1):
        rows = min(l, L + 1) if l > spin else 0  # orders that started below l
        if rows:
            den = torch.sqrt(((l * l - m * m) * (l * l - spin * spin)).clamp(min=0))
            A = math.sqrt((2 * l + 1.0) * (2 * l - 1)) * l / den
            B = A * m * spin / (l * (l - 1.0)) if l > 1 else torch.zeros_like(A)
            d1 = torch.sqrt((((l - 1) ** 2 - m * m) * ((l - 1) ** 2 - spin * spin)).clamp(min=0))
            C = math.sqrt((2 * l + 1) / max(2 * l - 3.0, 1.0)) * l * d1 / (max(l - 1, 1) * den)
            chains[0].step(rows, A, B, x, C)
            chains[1].step(rows, A, -B, x, C)
        if l % 16 == 0:
            chains[0].settle()
            chains[1].settle()
        rows = l + 1
        yield l, rows, chains[0].value(rows), chains[1].value(rows)


class _Torus:
    """Values of doubled ring functions at points (and the transpose), by FFT and Kaiser-Bessel gridding."""

    W, BETA = 16, 36.8

    def __init__(self, L, mm, M, pts):
        self.L, self.mm, self.M, self.n = L, mm, M, _good(max(4 * L + 4, 64))
        self.al = self.W * math.pi / self.n
        ks = torch.arange(-L, L + 1, dtype=torch.float64, device="cuda")

        def corr(k):
            s = torch.sqrt(self.BETA**2 - (k * self.al) ** 2)
            return (2 * math.pi / self.n) / (self.al * (torch.exp(s - self.BETA) - torch.exp(-s - self.BETA)) / s)

        self.dk, self.dm = corr(ks), corr(torch.arange(mm + 1, dtype=torch.float64, device="cuda"))
        self.kk = ks.long()
        self.pts = pts

    def _weights(self, t):
        t = torch.remainder(t, 2 * math.pi) * (self.n / (2 * math.pi))
        i0 = torch.ceil(t - self.W / 2)
        ws = []
        for j in range(self.W):
            z = (t - i0 - j) / (self.W / 2)
            r = self.BETA * torch.sqrt((1 - z * z).clamp(min=0))
            ws.append(torch.special.i0e(r) * torch.exp(r - self.BETA))
        return i0.long(), ws

    def _taps(self, lo, hi):
        i1, w1 = self._weights(self.pts[lo:hi, 0])
        i2, w2 = self._weights(self.pts[lo:hi, 1])
        for a in range(self.W):
            row = torch.remainder(i1 + a, self.n) * self.n
            for b in range(self.W):
                yield row + torch.remainder(i2 + b, self.n), w1[a] * w2[b]

    def spectrum(self, F, sgn):
        """c[m, k] of the ring functions F [m][M/2 + 1] doubled with the signs sgn[m]."""
        G = torch.cat([F, sgn[:, None] * F[:, 1:-1].flip(1)], dim=1)
        return torch.fft.fft(G, dim=1, norm="forward")[:, self.kk % self.M]

    def values(self, c):
        S = torch.zeros((self.n, self.mm + 1), dtype=torch.complex128, device="cuda")
        S[self.kk % self.n] = (c * self.dk * self.dm[:, None]).T
        g = torch.fft.irfft(torch.fft.ifft(S, dim=0, norm="forward"), n=self.n, dim=1, norm="forward").reshape(-1)
        del S
        out = torch.zeros(self.pts.shape[0], dtype=torch.float64, device="cuda")
        for lo in range(0, out.numel(), 1 << 23):
            hi = min(out.numel(), lo + (1 << 23))
            for i, w in self._taps(lo, hi):
                out[lo:hi].addcmul_(w, g[i])
        return out

    def rings(self, y, sgn):
        """The transpose: ring functions [m][M/2 + 1] from point values, folded with sgn[m]."""
        g = torch.zeros(self.n * self.n, dtype=torch.float64, device="cuda")
        for lo in range(0, y.numel(), 1 << 23):
            hi = min(y.numel(), lo + (1 << 23))
            for i, w in self._taps(lo, hi):
                g.index_add_(0, i, w * y[lo:hi])
        S = torch.fft.rfft(g.view(self.n, self.n), dim=1)[:, : self.mm + 1]
        c = torch.fft.fft(S, dim=0)[self.kk % self.n].T * self.dk * self.dm[:, None]
        H = torch.zeros((self.mm + 1, self.M), dtype=torch.complex128, device="cuda")
        H[:, self.kk % self.M] = c
        H = torch.fft.ifft(H, dim=1)
        h = self.M // 2
        F = H[:, : h + 1].clone()
        F[:, 1:h] += sgn[:, None] * H[:, h + 1 :].flip(1)
        return F


def _parity(mm, s=0):
    return 1.0 - 2.0 * (torch.arange(mm + 1, device="cuda", dtype=torch.float64) + s).remainder(2)


def _at(L, l, rows):
    m = torch.arange(rows, device="cuda")
    return m * (2 * L + 1 - m) // 2 + l


def _ring_sums(L, mm, M, a):
    a = a.to(torch.complex128).clone()
    a[: L + 1] = a[: L + 1].real + 0j
    fr, fi = (torch.zeros((mm + 1, M // 2 + 1), dtype=torch.float64, device="cuda") for _ in range(2))
    for l, rows, P in _legendre(L, mm, M):
        al = a[_at(L, l, rows)]
        fr[:rows].addcmul_(P, al.real[:, None])
        fi[:rows].addcmul_(P, al.imag[:, None])
    return torch.complex(fr, fi)


def _exact_torus(L, mm, pts):
    return _Torus(L, mm, _good(2 * L + 2), pts.double())


def _exact_spec(t, a):
    return t.spectrum(_ring_sums(t.L, t.mm, t.M, a), _parity(t.mm))


def _exact_adjoint(t, y, wpos=1.0):
    F = torch.view_as_real(t.rings(y.double(), _parity(t.mm)))
    out = torch.zeros(nu.nalm(t.L, t.mm), dtype=torch.complex128, device="cuda")
    for l, rows, P in _legendre(t.L, t.mm, t.M):
        out[_at(t.L, l, rows)] = torch.view_as_complex(torch.bmm(P[:, None, :], F[:rows])[:, 0, :].contiguous())
    out[: t.L + 1] = out[: t.L + 1].real + 0j
    out[t.L + 1 :] *= wpos
    return out


def _exact_grad(t, c):
    m = torch.arange(t.mm + 1, device="cuda", dtype=torch.float64)
    return t.values(c * (1j * t.kk.double())), t.values(c * (1j * m)[:, None])


def _exact_spin(case, s):
    L, sp = case["lmax"], case["spin"]
    t = _exact_torus(L, L, s["pts"])
    sg, sgn = (-1.0) ** sp, _parity(L, sp)
    G, C = s["a"].clone(), s["c"].clone()
    for v in (G, C):
        v[: L + 1] = v[: L + 1].real + 0j
    fq, fu = (torch.zeros((L + 1, t.M // 2 + 1), dtype=torch.complex128, device="cuda") for _ in range(2))
    hq, hu = (t.rings(s[k], sgn) for k in ("y", "u"))
    og, oc = (torch.zeros(nu.nalm(L), dtype=torch.complex128, device="cuda") for _ in range(2))
    for l, rows, p, n in _wigner(L, t.M, sp):
        i = _at(L, l, rows)
        w, x = 0.5 * (p + sg * n), 0.5 * (p - sg * n)
        g, c = G[i][:, None], C[i][:, None]
        fq[:rows] += g * w + 1j * c * x
        fu[:rows] += c * w - 1j * g * x
        og[i] = (w * hq[:rows] + 1j * x * hu[:rows]).sum(1)
        oc[i] = (w * hu[:rows] - 1j * x * hq[:rows]).sum(1)
    for v in (og, oc):
        v[: L + 1] = v[: L + 1].real + 0j
    return dict(q=t.values(t.spectrum(fq, sgn)), u=t.values(t.spectrum(fu, sgn)), g=og, c=oc)


def exact(case, seed):
    k = case["kind"]
    s = _inputs(case, seed)
    if k == "batch":
        out = dict(map=[], alm=[])
        for l, pts, a, y in s:
            t = _exact_torus(l, l, pts)
            out["map"].append(t.values(_exact_spec(t, a)))
            out["alm"].append(_exact_adjoint(t, y))
        return out
    if k == "spin":
        return _exact_spin(case, s)
    t = _exact_torus(case["lmax"], _mmax(case), s["pts"])
    if k == "synth":
        return t.values(_exact_spec(t, s["a"]))
    if k == "adjoint":
        return _exact_adjoint(t, s["y"])
    if k == "step":
        return dict(map=t.values(_exact_spec(t, s["a"])), alm=_exact_adjoint(t, s["y"]))
    if k == "pointing":
        dth, dph = _exact_grad(t, _exact_spec(t, s["phi"]))
        th, ph = s["pts"].unbind(1)
        return _shift(th, ph, dth, dph / torch.sin(th))
    c = _exact_spec(t, s["a"])
    f = t.values(c)
    g = 2 * s["w"].double() * f
    dth, dph = _exact_grad(t, c)
    return dict(map=f, grad_alm=_exact_adjoint(t, g, 2.0), grad_pts=torch.stack([g * dth, g * dph], 1))
