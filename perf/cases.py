"""The transforms a user of this library runs, for measuring: the cases, their inputs, one pass, and the exact answer.

A pass goes through the public binding (paper_1904_10514_gb300.Plan and the autograd
functions analyze / cl).  Kinds of pass:

  analysis   maps -> a_lm -> C_l, one nside for the whole batch (the main use)
  uneven     the same for maps of several nsides in one plan, replayed as a CUDA graph
  gradient   loss sum_l w_l (C_l - C*_l)^2, w_l = 1/l, and its gradient with respect to the maps
  synthesis  a_lm -> maps
  healpix    the equal-weight analysis with Jacobi steps that the method is compared with

Maps are Gaussian red-spectrum skies (power per degree l^-alpha, alpha in [1.5, 2.5]) plus
1e-3 white pixel noise, a_lm Gaussian with the same spectra: the inputs of the repository's
benchmark and tests.  They are made on the GPU from the seed alone.

exact() repeats each pass in float64 from the definitions: discrete Fourier sums per ring, the
unit-weight least squares in latitude, Gauss-Legendre projection on the normalised associated
Legendre functions (three-term recurrence with scaled start values).
"""

import math
from collections import OrderedDict

import numpy as np
import torch

import paper_1904_10514_gb300 as hp

DEV = "cuda"


# ---------------------------------------------------------------- the cases
def listed():
    return [
        # one small map in double precision, called on its own: latency and launches
        dict(name="analysis_fp64_n16", kind="analysis", nside=16, lmax=32, batch=1, precision="fp64"),
        # one ordinary map, single precision (a quick look at one sky)
        dict(name="analysis_n256", kind="analysis", nside=256, lmax=512, batch=1, precision="fp32"),
        # a handful of maps with a band limit below the grid's and of odd size
        dict(name="analysis_n128_l200_b5", kind="analysis", nside=128, lmax=200, batch=5, precision="fp32"),
        # the reference-precision form at a working resolution
        dict(name="analysis_fp64_n512", kind="analysis", nside=512, lmax=1024, batch=1, precision="fp64"),
        # a simulation ensemble: 64 maps at nside 512
        dict(name="analysis_n512_b64", kind="analysis", nside=512, lmax=1024, batch=64, precision="fp32"),
        # the benchmark batch: 32 maps at nside 1024
        dict(name="analysis_n1024_b32", kind="analysis", nside=1024, lmax=2048, batch=32, precision="fp32",
             autotune=True),
        # 200 maps of mixed resolution in one graph launch
        dict(name="uneven_200", kind="uneven", maps=200, largest=1024, mix=4000, precision="fp32"),
        # spectrum fitting: a C_l loss and its map gradient, a medium batch
        dict(name="gradient_n256_b16", kind="gradient", nside=256, lmax=512, batch=16, precision="fp32"),
        # the same at the largest grid
        dict(name="gradient_n2048_b8", kind="gradient", nside=2048, lmax=4096, batch=8, precision="fp32"),
        # simulating skies from coefficients
        dict(name="synthesis_n512_b32", kind="synthesis", nside=512, lmax=1024, batch=32, precision="fp32"),
        # a few skies at a time
        dict(name="synthesis_n256_l400_b6", kind="synthesis", nside=256, lmax=400, batch=6, precision="fp32"),
        # the comparison method with its usual three iterations
        dict(name="healpix_n256_b16", kind="healpix", nside=256, lmax=512, batch=16, precision="fp32", niter=3),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["analysis", "analysis", "analysis", "uneven", "gradient", "gradient", "synthesis", "healpix"])
    prec = "fp64" if kind != "uneven" and rng.random() < 0.25 else "fp32"
    if kind == "uneven":
        return dict(kind=kind, maps=_log_int(rng, 3, 200), largest=rng.choice([64, 128, 256, 512]),
                    mix=rng.randrange(1 << 20), precision=prec)
    nside = 2 ** rng.randint(3, 8 if prec == "fp64" else 9)
    # at most the pixels of 64 maps at nside 512 (double precision, and the iterated passes: a quarter)
    room = 64 * 512 * 512 // (nside * nside)
    if prec == "fp64" or kind == "healpix":
        room //= 4
    case = dict(kind=kind, nside=nside, lmax=2 * nside if rng.random() < 0.4 else rng.randint(nside // 2, 2 * nside),
                batch=_log_int(rng, 1, max(1, min(64, room))), precision=prec)
    if kind == "healpix":
        case["niter"] = rng.randint(0, 3)
    return case


def _nsides(case):
    """Nside of every map of an uneven batch: 64 .. `largest`, mostly small ones."""
    rng = np.random.Generator(np.random.PCG64(case["mix"]))
    sizes = [n for n in (64, 128, 256, 512, 1024) if n <= case["largest"]]
    p = np.array([0.40, 0.30, 0.15, 0.10, 0.05])[:len(sizes)]
    return [int(v) for v in rng.choice(sizes, size=case["maps"], p=p / p.sum())]


def _n_alm(L):
    return (L + 1) * (L + 2) // 2


def work(case):
    e = 8 if case["precision"] == "fp64" else 4
    if case["kind"] == "uneven":
        parts = [(n, 2 * n, 1) for n in _nsides(case)]
    else:
        parts = [(case["nside"], case["lmax"], case["batch"])]
    nbytes = flops = 0.0
    for nside, L, B in parts:
        maps, alm, cl = 12.0 * nside * nside * e, 2.0 * _n_alm(L) * e, 8.0 * (L + 1)
        # ring FFTs, one latitude FFT per order, and the sum over latitudes for every coefficient
        one = (2.5 * 12 * nside * nside * math.log2(4 * nside) + 5.0 * (L + 1) * 4 * nside * math.log2(4 * nside)
               + 4.0 * _n_alm(L) * (nside + 1))
        kind = case["kind"]
        if kind in ("analysis", "uneven"):
            nbytes += B * (maps + alm + cl)
            flops += B * one
        elif kind == "gradient":
            nbytes += B * (2 * maps + cl)
            flops += B * 2 * one
        elif kind == "synthesis":
            nbytes += B * (maps + alm)
            flops += B * one
        else:
            nbytes += B * (maps + alm)
            flops += B * one * (1 + 2 * case["niter"])
    return {"bytes": nbytes, "flops": flops}


# ---------------------------------------------------------------- inputs
_PLANS = OrderedDict()   # a program keeps the plan of its sizes; inputs change


def _plan(key, make):
    if key in _PLANS:
        _PLANS.move_to_end(key)
        return _PLANS[key]
    while _PLANS and sum(p.nbytes for p in _PLANS.values()) > 60e9:
        _PLANS.popitem(last=False)
    _PLANS[key] = make()
    return _PLANS[key]


def _plan_of(case):
    key = tuple(sorted((k, v) for k, v in case.items() if k not in ("name", "niter")))
    prec = case["precision"]
    if case["kind"] == "uneven":
        return _plan(key, lambda: hp.Plan(nsides=_nsides(case), precision=prec, graph=True))
    return _plan(key, lambda: hp.Plan(case["nside"], case["lmax"], case["batch"], prec,
                                      autotune=bool(case.get("autotune")), synthesis=case["kind"] == "synthesis",
                                      jacobi=case["kind"] == "healpix"))


def _rings(nside):
    """Per ring, north to south: cos(theta), sin(theta), points, first longitude, first pixel (numpy)."""
    j = np.arange(1, 4 * nside)
    cap = np.minimum(j, 4 * nside - j)
    polar = cap < nside
    half = np.where(polar, 1.0 - cap ** 2 / (3.0 * nside ** 2), 0.0)
    z = np.where(polar, np.where(j < 2 * nside, half, -half), 2.0 * (2 * nside - j) / (3.0 * nside))
    th = np.where(polar, 2.0 * np.arcsin(np.minimum(cap, nside) / (math.sqrt(6.0) * nside)), np.arccos(np.clip(z, -1, 1)))
    th = np.where(polar & (j > 2 * nside), np.pi - th, th)
    n = np.where(polar, 4 * cap, 4 * nside)
    phi0 = np.where(polar | (j % 2 == 0), np.pi / n, 0.0)
    start = np.concatenate([[0], np.cumsum(n)[:-1]])
    return th, n, phi0, start


def _skies(nside, batch, dtype, g, lmax):
    """`batch` red-spectrum maps: plane waves of log-spaced wavenumbers 2 .. lmax restricted to the sphere,
    amplitudes of a power law per map, plus white pixel noise."""
    K = 32
    th, n, phi0, start = _rings(nside)
    t = lambda a, d=torch.float32: torch.as_tensor(np.ascontiguousarray(a), device=DEV).to(d)  # noqa: E731
    k = torch.exp(torch.rand(K, generator=g, device=DEV) * math.log(max(2.0, lmax / 2.0))) * 2.0
    d = torch.randn(3, K, generator=g, device=DEV)
    wave = d / d.norm(dim=0, keepdim=True) * k
    alpha = 1.5 + torch.rand(batch, 1, generator=g, device=DEV)
    amp = torch.randn(2, batch, K, generator=g, device=DEV) * k ** ((2.0 - alpha) / 2) / math.sqrt(K)
    npix = 12 * nside * nside
    maps = torch.empty(batch, npix, dtype=dtype, device=DEV)
    ring = torch.repeat_interleave(torch.arange(len(n), device=DEV), t(n, torch.int64))
    step = 1 << 20
    for p0 in range(0, npix, step):
        r = ring[p0:p0 + step]
        i = torch.arange(p0, min(p0 + step, npix), device=DEV) - t(start, torch.int64)[r]
        phi = t(phi0)[r] + 2 * math.pi * i / t(n)[r]
        st, ct = torch.sin(t(th))[r], torch.cos(t(th))[r]
        arg = torch.stack([st * torch.cos(phi), st * torch.sin(phi), ct]).t() @ wave
        maps[:, p0:p0 + step] = (amp[0] @ torch.cos(arg).t() + amp[1] @ torch.sin(arg).t()).to(dtype)
    maps += 1e-3 * torch.randn(maps.shape, generator=g, device=DEV, dtype=dtype)
    return maps


def _coefficients(lmax, batch, dtype, g):
    """Gaussian a_lm, m-major, with <|a_lm|^2> = l^-alpha (zero below degree 2) and real a_l0."""
    m = torch.repeat_interleave(torch.arange(lmax + 1, device=DEV), lmax + 1 - torch.arange(lmax + 1, device=DEV))
    l = torch.arange(m.numel(), device=DEV) - (m * (2 * lmax + 1 - m)) // 2
    alpha = 1.5 + torch.rand(batch, 1, generator=g, device=DEV, dtype=dtype)
    sd = torch.where(l >= 2, l.clamp(min=2).to(dtype) ** (-alpha / 2), torch.zeros((), dtype=dtype, device=DEV))
    z = torch.randn(2, batch, m.numel(), generator=g, device=DEV, dtype=dtype) * math.sqrt(0.5)
    re = torch.where(m == 0, z[0] * math.sqrt(2.0), z[0])
    return torch.complex(sd * re, sd * torch.where(m == 0, torch.zeros_like(z[1]), z[1]))


def _gen(seed):
    g = torch.Generator(device=DEV)
    g.manual_seed(int(seed))
    return g


def _target(L, g):
    """w_l = 1 / l (l >= 2) and a seeded power law C*_l."""
    l = torch.arange(L + 1, device=DEV, dtype=torch.float64)
    w = torch.where(l >= 2, 1.0 / l.clamp(min=1), 0.0)
    c = torch.where(l >= 2, l.clamp(min=2) ** -2.0, 0.0)
    return w, c * (0.5 + torch.rand(L + 1, generator=g, device=DEV, dtype=torch.float64))


def _inputs(case, seed):
    g = _gen(seed)
    dt = torch.float64 if case["precision"] == "fp64" else torch.float32
    s = {}
    if case["kind"] == "uneven":
        ns = _nsides(case)
        pieces = {n: iter(_skies(n, ns.count(n), dt, g, 2 * n)) for n in sorted(set(ns))}
        s["maps"] = torch.cat([next(pieces[n]) for n in ns])
    elif case["kind"] == "synthesis":
        s["alm"] = _coefficients(case["lmax"], case["batch"], dt, g)
    else:
        s["maps"] = _skies(case["nside"], case["batch"], dt, g, case["lmax"])
    if case["kind"] == "gradient":
        s["w"], s["target"] = _target(case["lmax"], g)
    return s


def prepare(case, seed):
    s = _inputs(case, seed)
    s["plan"] = _plan_of(case)
    s["kind"] = case["kind"]
    if case["kind"] == "uneven":   # a graph is replayed on fixed buffers
        s["alm"] = torch.empty(s["plan"].nalm, dtype=s["plan"].cdtype, device=DEV)
        s["cl"] = torch.empty(s["plan"].ncl, dtype=torch.float64, device=DEV)
    elif case["kind"] == "gradient":
        s["maps"].requires_grad_(True)
    elif case["kind"] == "healpix":
        s["niter"] = case["niter"]
    return s


def run(s):
    plan, kind = s["plan"], s["kind"]
    if kind == "analysis":
        alm = plan.analyze(s["maps"])
        return {"alm": alm, "cl": plan.cl(alm)}
    if kind == "uneven":
        plan.analyze(s["maps"], out=s["alm"])
        plan.cl(s["alm"], out=s["cl"])
        return {"alm": s["alm"], "cl": s["cl"]}
    if kind == "gradient":
        cl = hp.cl(hp.analyze(s["maps"], plan), plan)
        loss = torch.sum(s["w"] * (cl - s["target"]) ** 2)
        (grad,) = torch.autograd.grad(loss, s["maps"])
        return {"cl": cl.detach(), "grad": grad}
    if kind == "synthesis":
        return {"maps": plan.sh_synthesis(s["alm"])}
    return {"alm": plan.healpix_analysis(s["maps"], niter=s["niter"])}


# ---------------------------------------------------------------- the same in 64 bits
F64 = torch.float64


def _legendre(theta, L, lb=16):
    """Blocks of orthonormal Pbar_l^m(cos theta), Condon-Shortley phase: (first degree, P[m, l, node]).  Values are
    kept as p 2^(-600 e) so that the start values sin^m(theta) do not underflow."""
    x, st = torch.cos(theta), torch.sin(theta)
    N = theta.numel()
    m = torch.arange(L + 1, device=DEV, dtype=F64)
    cur, prev = (torch.zeros(L + 1, N, dtype=F64, device=DEV) for _ in range(2))
    ex = torch.zeros(L + 1, N, dtype=torch.int32, device=DEV)
    top, top_e = torch.full((N,), math.sqrt(0.5), dtype=F64, device=DEV), torch.zeros(N, dtype=torch.int32, device=DEV)
    for l0 in range(0, L + 1, lb):
        l1 = min(L + 1, l0 + lb)
        P = torch.zeros(L + 1, l1 - l0, N, dtype=F64, device=DEV)
        for l in range(l0, l1):
            if l > 0:
                mm = m[:l, None]
                a = torch.sqrt((4.0 * l * l - 1.0) / (float(l) * l - mm * mm))
                b = torch.sqrt(((l - 1.0) ** 2 - mm * mm).clamp(min=0.0) / max(4.0 * (l - 1.0) ** 2 - 1.0, 1.0))
                new = a * (x * cur[:l] - b * prev[:l])
                prev[:l], cur[:l] = cur[:l], new
                top = top * st * -math.sqrt((2 * l + 1.0) / (2 * l))
                small = top.abs() < 2.0 ** -300
                top = torch.where(small & (top != 0), top * 2.0 ** 600, top)
                top_e = top_e + (small & (top != 0)).int()
            cur[l], ex[l] = top, top_e
            P[:l + 1, l - l0] = torch.where(ex[:l + 1] == 0, cur[:l + 1], 0.0)
        big = (cur.abs() > 2.0 ** 250) & (ex > 0)
        f = torch.where(big, torch.full_like(cur, 2.0 ** -600), torch.ones_like(cur))
        cur, prev, ex = cur * f, prev * f, ex - big.int()
        yield l0, P


def _project(Z, theta, L):
    """a[m, l, :] = sum over the half nodes of Pbar_l^m Z[m parity][symmetry][m, node, :]."""
    A = torch.zeros(L + 1, L + 1, Z[0][0].shape[-1], dtype=F64, device=DEV)
    for l0, P in _legendre(theta, L):
        lb = P.shape[1]
        for mp in range(min(2, L + 1)):
            for s in range(2):
                off = (l0 ^ mp ^ s) & 1
                k = (min(L, l0 + lb - 1) - mp) // 2 + 1
                if off < lb and k > 0:
                    A[mp::2, l0 + off:l0 + lb:2][:k] = torch.bmm(P[mp::2, off::2][:k], Z[mp][s][:k])
    return A


def _expand(A, theta, L):
    """The transpose of _project: Z[m parity][symmetry][m, node, :]."""
    N, C = theta.numel(), A.shape[-1]
    Z = [[torch.zeros((L - mp) // 2 + 1 if L >= mp else 0, N, C, dtype=F64, device=DEV) for _ in range(2)]
         for mp in range(2)]
    for l0, P in _legendre(theta, L):
        lb = P.shape[1]
        for mp in range(min(2, L + 1)):
            for s in range(2):
                off = (l0 ^ mp ^ s) & 1
                k = (min(L, l0 + lb - 1) - mp) // 2 + 1
                if off < lb and k > 0:
                    Z[mp][s][:k] += torch.bmm(P[mp::2, off::2][:k].transpose(1, 2), A[mp::2, l0 + off:l0 + lb:2][:k])
    return Z


def _gauss(n):
    """Positive half of the n-point Gauss-Legendre rule (n even): theta, weights.  Newton in theta, P_n by the
    recurrence for P_k - P_(k-1) in 1 - cos(theta) = 2 sin^2(theta / 2), which keeps its digits near theta = 0."""
    t = np.pi * (np.arange(n // 2) + 0.75) / (n + 0.5)
    for _ in range(5):
        y = 2.0 * np.sin(t / 2) ** 2
        p, d = 1.0 - y, -y
        before = np.ones_like(t)
        for k in range(2, n + 1):
            d = ((k - 1) * d - (2 * k - 1) * y * p) / k
            before, p = p, p + d
        slope = -n * (before - (1.0 - y) * p) / np.sin(t)   # d P_n / d theta
        t = t - p / slope
    at = lambda a: torch.as_tensor(a, device=DEV, dtype=F64)  # noqa: E731
    return at(t), at(2.0 / slope ** 2)


def _pack(A, L):
    """a[m, l, 2B] -> (B, n_alm) complex, and back."""
    m, l = torch.triu_indices(L + 1, L + 1, device=DEV)
    return torch.view_as_complex(A[m, l].view(m.numel(), -1, 2)).t().contiguous()


def _unpack(a, L):
    m, l = torch.triu_indices(L + 1, L + 1, device=DEV)
    A = torch.zeros(L + 1, L + 1, 2 * a.shape[0], dtype=F64, device=DEV)
    A[m, l] = torch.view_as_real(a.t().contiguous()).reshape(m.numel(), -1)
    return A


def _columns(y):
    """(B, R, L+1) complex -> [m, R, 2B] real."""
    return torch.view_as_real(y.permute(2, 1, 0).contiguous()).flatten(2)


def _uncolumns(Y):
    return torch.view_as_complex(Y.unflatten(2, (-1, 2)).contiguous()).permute(2, 1, 0)


class _Grid:
    def __init__(self, nside, L):
        self.nside, self.L, self.p = nside, L, 2 * nside
        th, n, phi0, start = _rings(nside)
        self.n, self.phi0, self.start = n, phi0, start
        self.theta = torch.as_tensor(th, device=DEV, dtype=F64)
        self.sign = (1.0, -1.0)

    def ring_groups(self):
        """(ring indices, points): the polar rings in pairs, the equatorial ones together."""
        N = self.nside
        for i in range(N - 1):
            yield [i, 4 * N - 2 - i], int(self.n[i])
        yield list(range(N - 1, 3 * N)), 4 * N

    def gather(self, f, rows, n):
        if len(rows) == 2 and n < 4 * self.nside:
            return torch.stack([f[:, self.start[r]:self.start[r] + n] for r in rows], 1)
        return f[:, self.start[rows[0]]:self.start[rows[0]] + len(rows) * n].view(f.shape[0], len(rows), n)

    def phase(self, rows, m):
        """e^{-i m phi0} per ring and order, m phi0 reduced modulo 2 pi exactly."""
        n = torch.as_tensor(self.n[rows], device=DEV)[:, None]
        sh = torch.as_tensor(self.phi0[rows] > 0, device=DEV)[:, None]
        r = torch.where(sh, m[None] % (2 * n), torch.zeros_like(m[None] % (2 * n)))
        return torch.polar(torch.ones_like(r, dtype=F64), -math.pi * r.to(F64) / n)

    # step 1 of the method: ring interpolants at un-shifted longitudes, pole values
    def interp_weights(self, rows, n):
        h = n // 2
        m = torch.arange(min(h, self.L) + 1, device=DEV)
        w = self.phase(rows, m) / n
        if h <= self.L:
            half = 0.5 * w[:, h]
            w[:, h] = half if h < self.p else half.real.to(w.dtype)
        return w

    def poles(self):
        N = self.nside
        xs, ys, pn, ps = [], [], [], []
        for i in range(3):
            lam = self.phi0[i] + 2 * np.pi * np.arange(self.n[i]) / self.n[i]
            s = math.sin(float(self.theta[i]))
            xs.append(s * np.cos(lam))
            ys.append(s * np.sin(lam))
            pn.append(self.start[i] + np.arange(self.n[i]))
            ps.append(self.start[4 * N - 2 - i] + np.arange(self.n[i]))
        scale = math.sin(float(self.theta[2]))   # the constant term does not depend on the unit of length
        x, y = np.concatenate(xs) / scale, np.concatenate(ys) / scale
        w = np.linalg.pinv(np.stack([np.ones_like(x), x, y, x * x, x * y, y * y], 1))[0]
        t = lambda a: torch.as_tensor(np.concatenate(a), device=DEV)  # noqa: E731
        return t(pn), t(ps), torch.as_tensor(w, device=DEV)

    def latitude_rows(self, f):
        y = torch.zeros(f.shape[0], 4 * self.nside + 1, self.L + 1, dtype=torch.complex128, device=DEV)
        for rows, n in self.ring_groups():
            w = self.interp_weights(rows, n)
            c = torch.fft.rfft(self.gather(f, rows, n), dim=-1)[..., :w.shape[1]] * w
            y[:, torch.as_tensor(rows, device=DEV) + 1, :w.shape[1]] = c
        pn, ps, w = self.poles()
        y[:, 0, 0], y[:, -1, 0] = (f[:, pn] @ w).to(y.dtype), (f[:, ps] @ w).to(y.dtype)
        return y

    def latitude_rows_t(self, gy):
        g = torch.zeros(gy.shape[0], 12 * self.nside ** 2, dtype=F64, device=DEV)
        for rows, n in self.ring_groups():
            w = self.interp_weights(rows, n)
            s = torch.zeros(gy.shape[0], len(rows), n, dtype=torch.complex128, device=DEV)
            s[..., :w.shape[1]] = gy[:, torch.as_tensor(rows, device=DEV) + 1, :w.shape[1]].conj() * w
            self.gather(g, rows, n)
            v = torch.fft.fft(s, dim=-1).real
            for q, r in enumerate(rows):
                g[:, self.start[r]:self.start[r] + n] = v[:, q]
        pn, ps, w = self.poles()
        g[:, pn] += gy[:, 0, 0].real[:, None] * w
        g[:, ps] += gy[:, -1, 0].real[:, None] * w
        return g

    # steps 2 and 3: least squares in latitude, evaluation at the Gauss nodes
    def solver(self):
        N, p = self.nside, self.p
        self.gt, gw = _gauss(p + 2)
        th = torch.cat([torch.zeros(1, dtype=F64, device=DEV), self.theta[:2 * N]])
        th[-1] = math.pi / 2
        w = torch.full_like(th, 2.0)
        w[0] = 1.0
        pair = 2.0 * w
        pair[-1] = 2.0
        G = [[None, None], [None, None]]
        for mp in range(2):
            for s in range(2):
                j = torch.arange((mp + s) % 2, p + 1, 2, device=DEV, dtype=F64)
                if mp == 1 and s == 1:
                    j = j[1:]
                fn = torch.sin if mp else torch.cos
                B = fn(th[:, None] * j)
                T = B.t() @ (pair[:, None] * B)
                X = torch.cholesky_solve((w[:, None] * B).t(), torch.linalg.cholesky(T))
                G[mp][s] = (2.0 * math.sqrt(2 * math.pi) * gw[:, None]) * (fn(self.gt[:, None] * j) @ X)
        return G

    def fold(self, Y):
        """[m, Q, C] -> symmetric and antisymmetric halves [m, 2 Nside + 1, C]."""
        h = Y.shape[1] // 2
        out = []
        for sg in self.sign:
            v = Y[:, :h + 1].clone()
            v[:, :h] += sg * Y[:, h + 1:].flip(1)
            out.append(v)
        return out

    def analysis(self, f):
        G = self.solver()
        Z = [[G[mp][s] @ v for s, v in enumerate(self.fold(_columns(self.latitude_rows(f)[..., mp::2])))]
             for mp in range(2)]
        return _pack(_project(Z, self.gt, self.L), self.L)

    def analysis_t(self, ga):
        G = self.solver()
        Z = _expand(_unpack(ga, self.L), self.gt, self.L)
        gy = torch.zeros(ga.shape[0], 4 * self.nside + 1, self.L + 1, dtype=torch.complex128, device=DEV)
        for mp in range(2):
            if mp > self.L:
                continue
            a, b = (G[mp][s].t() @ Z[mp][s] for s in range(2))
            Y = torch.cat([a + b, (a - b)[:, :-1].flip(1)], 1)
            Y[:, a.shape[1] - 1] = a[:, -1] + b[:, -1]
            gy[..., mp::2] = _uncolumns(Y)
        return self.latitude_rows_t(gy)

    # the synthesis at the pixel centres and its transpose
    def synthesis(self, a):
        N, L, B = self.nside, self.L, a.shape[0]
        a = a.clone()
        a[:, :L + 1] = a[:, :L + 1].real.to(a.dtype)
        Z = _expand(_unpack(a, L), self.theta[:2 * N], L)
        F = torch.zeros(B, 4 * N - 1, L + 1, dtype=torch.complex128, device=DEV)
        for mp in range(min(2, L + 1)):
            nn, ss = Z[mp][0] + Z[mp][1], Z[mp][0] - Z[mp][1]
            F[..., mp::2] = _uncolumns(torch.cat([nn, ss[:, :-1].flip(1)], 1)) / math.sqrt(2 * math.pi)
        f = torch.empty(B, 12 * N * N, dtype=F64, device=DEV)
        m = torch.arange(L + 1, device=DEV)
        F[..., 1:] *= 2.0
        for rows, n in self.ring_groups():
            v = F[:, rows] * self.phase(rows, m).conj()
            k = m % n
            s = torch.zeros(B, len(rows), n, dtype=torch.complex128, device=DEV).index_add_(2, k, v)
            v = torch.fft.ifft(s, dim=-1).real * n
            for q, r in enumerate(rows):
                f[:, self.start[r]:self.start[r] + n] = v[:, q]
        return f

    def synthesis_t(self, f):
        N, L, B = self.nside, self.L, f.shape[0]
        m = torch.arange(L + 1, device=DEV)
        D = torch.empty(B, 4 * N - 1, L + 1, dtype=torch.complex128, device=DEV)
        for rows, n in self.ring_groups():
            D[:, rows] = torch.fft.fft(self.gather(f, rows, n), dim=-1)[..., m % n] * self.phase(rows, m)
        h, Z = 2 * N - 1, [[None, None], [None, None]]
        for mp in range(2):
            Y = _columns(D[..., mp::2]) / math.sqrt(2 * math.pi)
            for s, sg in enumerate(self.sign):
                v = Y[:, :h + 1].clone()
                v[:, :h] += sg * Y[:, h + 1:].flip(1)
                if s == 1:
                    v[:, h] = 0.0
                Z[mp][s] = v
        return _pack(_project(Z, self.theta[:2 * N], L), L)


def _cl(a, L):
    A = _unpack(a, L)   # [m, l, 2B]
    e = A.square().unflatten(2, (-1, 2)).sum(-1)
    e[1:] *= 2.0
    return (e.sum(0) / (2.0 * torch.arange(L + 1, device=DEV, dtype=F64)[:, None] + 1.0)).t().contiguous()


def exact(case, seed):
    s = _inputs(case, seed)
    kind = case["kind"]
    if kind == "uneven":
        ns, at, parts = _nsides(case), 0, {}
        for n in ns:
            parts.setdefault(n, []).append(s["maps"][at:at + 12 * n * n].double())
            at += 12 * n * n
        done = {}
        for n, v in parts.items():
            a = _Grid(n, 2 * n).analysis(torch.stack(v))
            done[n] = (iter(a), iter(_cl(a, 2 * n)))
        pairs = [[next(it) for it in done[n]] for n in ns]
        return {"alm": torch.cat([a for a, _ in pairs]), "cl": torch.cat([c for _, c in pairs])}
    L, grid = case["lmax"], _Grid(case["nside"], case["lmax"])
    if kind == "synthesis":
        return {"maps": grid.synthesis(s["alm"].to(torch.complex128))}
    f = s["maps"].double()
    if kind == "healpix":
        scale = 4.0 * math.pi / (12 * case["nside"] ** 2)
        a = scale * grid.synthesis_t(f)
        for _ in range(case["niter"]):
            a = a + scale * grid.synthesis_t(f - grid.synthesis(a))
        return {"alm": a}
    a = grid.analysis(f)
    cl = _cl(a, L)
    if kind == "analysis":
        return {"alm": a, "cl": cl}
    m, l = torch.triu_indices(L + 1, L + 1, device=DEV)
    gcl = 2.0 * s["w"] * (cl - s["target"])
    w = torch.where(m == 0, 2.0, 4.0).to(F64) / (2 * l + 1).to(F64)
    return {"cl": cl, "grad": grid.analysis_t(gcl[:, l] * w * a)}
