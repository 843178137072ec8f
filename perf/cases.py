"""Work that users of the wavelet transform have it do, as timed cases.

A case is one configuration and one call (or the analysis + synthesis pair) of
the Python binding.  Sizes are those of the repository's own workloads: the
headline configuration (L = 1024, N = 5, lambda = 2), the served mix (L =
round(exp U[ln 32, ln 2048]), N 1..8, lambda 2 or 3: most L are no power of
two), the batch of 64 signals with L in {64, 128, 256, 512}, and the
multi-resolution, McEwen-Wiaux-grid, harmonic-transform and FP64 paths.

``exact`` evaluates the same definitions (McEwen, Vandergheynst & Wiaux 2013)
in float64 with torch alone: Wigner functions by the three-term recurrence in
l, dense beta sums, torch FFTs in alpha.
"""
import math

import numpy as np
import torch

from paper_1308_5706_gb300 import binding as B

DEV = "cuda"


# ---- the cases ---------------------------------------------------------------

def _case(name, op, L, N, lam=2.0, J0=0, precision="mixed", grid="dh", signals=1):
    return {"name": name, "op": op, "L": L, "N": N, "lam": lam, "J0": J0, "precision": precision, "grid": grid,
            "signals": signals}


def listed():
    return [
        # the smallest served request: latency and launches count
        _case("ana_L32_N3", "analysis", 32, 3),
        # a small synthesis (a thresholded low-resolution map going back to f_lm)
        _case("syn_L128_N5", "synthesis", 128, 5),
        # served requests of the mixed load: ragged band-limits, another dilation, more orientations
        _case("ana_L361_N4_lam3", "analysis", 361, 4, 3.0, 1),
        _case("syn_L723_N6", "synthesis", 723, 6),
        # the headline configuration, each direction
        _case("ana_L1024_N5", "analysis", 1024, 5),
        _case("syn_L1024_N5", "synthesis", 1024, 5),
        # the largest transform the library takes
        _case("ana_L2048_N8", "analysis", 2048, 8),
        # every scale on the grid of its own band-limit: compression and denoising pipelines
        _case("multires_rt_L1024_N5", "roundtrip", 1024, 5, grid="multires"),
        # half the beta samples (McEwen-Wiaux grid), an odd band-limit
        _case("mw_rt_L511_N3", "roundtrip", 511, 3, grid="mw"),
        # pixels to harmonic coefficients and back
        _case("sht_rt_L1024", "sht", 1024, 1),
        # the float64 path, the paper's N = 3 experiment
        _case("fp64_rt_L512_N3", "roundtrip", 512, 3, precision="fp64"),
        # many signals per launch set: L in {64, 128, 256, 512}, N in {1, 3, 5}
        _case("batch_rt_64", "batch", 512, 5, signals=64),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """One more case: L over the logarithm of its range, every N, both dilations."""
    kind = rng.choice(["analysis", "synthesis", "analysis", "synthesis", "multires", "mw", "sht", "fp64", "batch"])
    lam, N = rng.choice([2.0, 2.0, 3.0]), rng.randint(1, 8)
    J0 = rng.choice([0, 0, 1, 2])
    op, grid, precision, signals = kind, "dh", "mixed", 1
    if kind in ("analysis", "synthesis"):
        L = _log_int(rng, 32, 2048)
    elif kind in ("multires", "mw"):
        op, grid, L = "roundtrip", kind, _log_int(rng, 32, 1300)
    elif kind == "sht":
        L, N, lam, J0 = _log_int(rng, 32, 2048), 1, 2.0, 0
    elif kind == "fp64":
        op, precision, L = "roundtrip", "fp64", _log_int(rng, 32, 512)
    else:
        L, N, lam, J0, signals = 64 << rng.randint(0, 3), 5, 2.0, 0, rng.randint(4, 64)
    c = _case("", op, L, N, lam, J0, precision, grid, signals)
    del c["name"]
    return c


# ---- inputs ------------------------------------------------------------------

def _signal(L, gen, dtype):
    """Harmonic coefficients of a real Gaussian field with C_l = 1/(l(l+1))
    (l >= 2), flat index l*l + l + m: f_{l,-m} = (-1)^m conj(f_lm)."""
    k = torch.arange(L * L, device=DEV)
    l = torch.sqrt(k.double()).long()
    l -= (l * l > k).long()
    l += ((l + 1) * (l + 1) <= k).long()
    m = k - l * l - l
    sd = torch.where(l >= 2, 1.0 / torch.sqrt((l * (l + 1)).double().clamp(min=1.0)), torch.zeros((), device=DEV))
    z = torch.view_as_complex(torch.randn(L * L, 2, generator=gen, device=DEV, dtype=torch.float64)) / math.sqrt(2.0)
    z = torch.where(m == 0, (z.real * math.sqrt(2.0)).to(z.dtype), z) * sd
    sgn = torch.where((m & 1) == 1, -1.0, 1.0)
    return torch.where(m < 0, sgn * z[l * l + l - m].conj(), z).to(dtype)


def _gen(seed):
    g = torch.Generator(device=DEV)
    g.manual_seed(int(seed))
    return g


def _dtypes(case):
    return (torch.complex128, torch.float64) if case["precision"] == "fp64" else (torch.complex64, torch.float32)


def _batch_config(case):
    """Band-limit and orientations of each signal of a batch (fixed mix)."""
    r = np.random.RandomState(case["signals"])
    top = int(round(math.log2(case["L"] / 64))) + 1
    return [(64 << int(a), (1, 3, 5)[int(b)]) for a, b in zip(r.randint(0, top, case["signals"]),
                                                             r.randint(0, 3, case["signals"]))]


def _up(n):
    return (n + 63) // 64 * 64  # buffers start on 256-byte boundaries


def prepare(case, seed):
    L, N = case["L"], case["N"]
    cd, rd = _dtypes(case)
    gen = _gen(seed)
    op = case["op"]
    if op == "batch":
        cfg = _batch_config(case)
        plans = [B.Plan(a, b, case["lam"], case["J0"], case["precision"]) for a, b in cfg]
        f, W, P, g = [], [], [], []
        sizes = [(_up(p.L * p.L), _up(math.prod(p.w_shape)), _up(math.prod(p.wphi_shape))) for p in plans]
        fb, gb = (torch.zeros(sum(s[0] for s in sizes), dtype=cd, device=DEV) for _ in range(2))
        Wb = torch.zeros(sum(s[1] for s in sizes), dtype=rd, device=DEV)
        Pb = torch.zeros(sum(s[2] for s in sizes), dtype=rd, device=DEV)
        of = ow = op_ = 0
        for p, s in zip(plans, sizes):
            f.append(fb[of:of + p.L * p.L])
            f[-1].copy_(_signal(p.L, gen, cd))
            g.append(gb[of:of + p.L * p.L])
            W.append(Wb[ow:ow + math.prod(p.w_shape)])
            P.append(Pb[op_:op_ + math.prod(p.wphi_shape)])
            of, ow, op_ = of + s[0], ow + s[1], op_ + s[2]
        return {"op": op, "plans": plans, "handles": [p.handle for p in plans], "f": f, "W": W, "Wphi": P, "g": g,
                "all": (Wb, Pb, gb)}
    plan = B.Plan(L, N, case["lam"], case["J0"], case["precision"], multires=case["grid"] == "multires",
                  mw=case["grid"] == "mw")
    s = {"op": op, "plan": plan}
    if op == "sht":
        s["f"], s["pix"], s["g"] = _signal(L, gen, cd), plan.alloc_pix(), plan.alloc_flm()
        return s
    if op == "synthesis":
        # coefficients after a pointwise operation (a threshold): no longer those of a band-limited signal
        s["W"] = torch.randn(plan.w_shape, generator=gen, device=DEV, dtype=rd)
        s["Wphi"] = torch.randn(plan.wphi_shape, generator=gen, device=DEV, dtype=rd)
    else:
        s["f"] = _signal(L, gen, cd)
        s["W"], s["Wphi"] = plan.alloc_w()
    if op != "analysis":
        s["g"] = plan.alloc_flm()
    return s


def run(s):
    op = s["op"]
    if op == "batch":
        B.s2dw_analysis_batch(s["handles"], s["f"], s["W"], s["Wphi"])
        B.s2dw_synthesis_batch(s["handles"], s["W"], s["Wphi"], s["g"])
        return s["all"]
    p = s["plan"]
    if op == "sht":
        p.sht_inverse(s["f"], s["pix"])
        p.sht_forward(s["pix"], s["g"])
        return s["pix"], s["g"]
    if op == "analysis":
        p.analysis(s["f"], s["W"], s["Wphi"])
        return s["W"], s["Wphi"]
    if op == "synthesis":
        p.synthesis(s["W"], s["Wphi"], s["g"])
        return s["g"]
    p.analysis(s["f"], s["W"], s["Wphi"])
    p.synthesis(s["W"], s["Wphi"], s["g"])
    return s["W"], s["Wphi"], s["g"]


# ---- scales, bands and the work of a pass ------------------------------------

def _j_max(L, lam):
    J, p = 0, 1.0
    while p < L:
        p *= lam
        J += 1
    return J


_GLX, _GLW = np.polynomial.legendre.leggauss(24)


def _bump_integral(lo, hi, lam):
    """int_lo^hi s_lambda(u)^2 / u du, limits clipped to [1/lambda, 1] (arrays)."""
    lo, hi = np.clip(lo, 1.0 / lam, 1.0), np.clip(hi, 1.0 / lam, 1.0)
    panels = 48
    h = (hi - lo) / panels
    u = lo[..., None, None] + h[..., None, None] * (np.arange(panels)[:, None] + 0.5 + 0.5 * _GLX)
    x = 2.0 * lam / (lam - 1.0) * (u - 1.0 / lam) - 1.0
    inside = np.abs(x) < 1.0
    v = np.where(inside, np.exp(-2.0 / np.where(inside, 1.0 - x * x, 1.0)), 0.0) / u
    return np.maximum((v * _GLW).sum((-1, -2)) * 0.5 * h, 0.0)


def _radial(L, lam, J0):
    """kappa^j(l) [J+1][L] and Phi_l [L]."""
    J = _j_max(L, lam) - J0
    l = np.arange(L)
    norm = _bump_integral(np.array(1.0 / lam), np.array(1.0), lam)
    t = lam ** np.arange(J + 1)[:, None] * l / L
    kap = np.sqrt(_bump_integral(t / lam, t, lam) / norm)
    tp = lam ** J * l / L
    return kap, np.sqrt(np.where(tp <= 1.0 / lam, 1.0, _bump_integral(tp, np.ones(L), lam) / norm))


def _direction(L, N):
    """s_{l n_k} [L][N], n_k = -(N-1) + 2k."""
    s = np.zeros((L, N), dtype=np.complex128)
    eta = 1.0 if N % 2 == 1 else 1j
    for l in range(1, L):
        g = min(N - 1, l - (1 + (-1) ** (N + l)) // 2)
        for k in range(N):
            n = -(N - 1) + 2 * k
            if (g - n) % 2 == 0 and 0 <= (g - n) // 2 <= g:
                s[l, k] = eta * math.sqrt(2.0 ** (-g) * math.comb(g, (g - n) // 2))
    return s


def _bands(kap, phi):
    hi = [int(np.nonzero(k > 0)[0][-1]) + 1 if (k > 0).any() else 0 for k in kap]
    return hi, int(np.nonzero(phi > 0)[0][-1]) + 1


def _one_work(L, N, lam, J0, grid, el):
    """Bytes of f and W, and flops of one direction: per triple (l, m', m) of
    the l-contraction a product with f and a complex-by-real multiply-add for
    each order, then one FFT per column in beta and per row in alpha."""
    kap, phi = _radial(L, lam, J0)
    bands, bphi = _bands(kap, phi)
    flops = samples = 0.0
    for j in range(len(bands) + 1):
        wav = j < len(bands)
        Lj, Nj, w = (bands[j], N, kap[j]) if wav else (bphi, 1, phi)
        lg = max(1, Lj) if grid == "multires" else L
        nb, n = (lg if grid == "mw" else 2 * lg), 2 * lg - 1
        l = np.nonzero(w > 0)[0].astype(np.float64)
        flops += float(((l + 1) ** 2).sum()) * (2 + 4 * Nj)
        flops += Nj * Lj * 5.0 * (2 * lg) * math.log2(2 * lg) + Nj * nb * 2.5 * n * math.log2(max(2, n))
        samples += Nj * nb * n
    return L * L * 2.0 * el + samples * el, flops


def work(case):
    el = 8 if case["precision"] == "fp64" else 4
    L, op = case["L"], case["op"]
    if op == "sht":
        l = np.arange(L) + 1.0
        flops = 2 * (6 * float((l ** 2).sum()) + L * 5.0 * 2 * L * math.log2(2 * L) + 2 * L * 2.5 * 2 * L * math.log2(2 * L))
        return {"bytes": 2.0 * (2 * L * L * el + 2 * L * (2 * L - 1) * el), "flops": flops}
    if op == "batch":
        parts = [_one_work(a, b, case["lam"], case["J0"], "dh", el) for a, b in _batch_config(case)]
        return {"bytes": 2.0 * sum(p[0] for p in parts), "flops": 2.0 * sum(p[1] for p in parts)}
    b, fl = _one_work(L, case["N"], case["lam"], case["J0"], case["grid"], el)
    k = 2.0 if op == "roundtrip" else 1.0
    return {"bytes": k * b, "flops": k * fl}


# ---- float64 evaluation of the definitions -----------------------------------

class _Wigner:
    """Delta^l_{m'm} = d^l_{m'm}(pi/2), 0 <= m', m <= l, l = 0, 1, ... in turn:
    the three-term recurrence in l on values scaled by 2^E (the first ones
    lie below the float64 range for l > 1000)."""

    def __init__(self, L):
        self.L, self.l = L, -1
        i = torch.arange(L, device=DEV, dtype=torch.float64)
        self.mp, self.m = i[:, None], i[None, :]
        self.cur = torch.zeros(L, L, device=DEV, dtype=torch.float64)
        self.old = torch.zeros_like(self.cur)
        self.E = torch.zeros_like(self.cur)

    def step(self):
        self.l += 1
        l, n = self.l, self.l + 1
        if l > 0:
            q = l - 1
            a = torch.sqrt((l * l - self.mp[:l] ** 2) * (l * l - self.m[:, :l] ** 2))
            b = torch.sqrt(((q * q - self.mp[:l] ** 2) * (q * q - self.m[:, :l] ** 2)).clamp(min=0.0))
            cur, old = self.cur[:l, :l], self.old[:l, :l]
            if q == 0:
                new = torch.zeros(1, 1, device=DEV, dtype=torch.float64)  # d^1_00(pi/2) = cos(pi/2)
            else:
                new = (-(2 * q + 1.0) * self.mp[:l] * self.m[:, :l] * cur - (q + 1.0) * b * old) / (q * a)
            self.old[:l, :l] = cur
            self.cur[:l, :l] = new
            big = self.cur[:l, :l].abs() > 1e120
            down = torch.tensor(2.0 ** -400, device=DEV, dtype=torch.float64)
            self.cur[:l, :l] = torch.where(big, self.cur[:l, :l] * down, self.cur[:l, :l])
            self.old[:l, :l] = torch.where(big, self.old[:l, :l] * down, self.old[:l, :l])
            self.E[:l, :l] += 400.0 * big
        # edge m' = l: (-1)^(l-m) sqrt(C(2l, l+m)) 2^-l, by the ratio of neighbours from m = l down
        r = np.ones(n)
        m = np.arange(l, 0, -1)
        r[1:] = np.sqrt((l + m) / (l - m + 1.0))
        mant, E = np.empty(n), np.empty(n)
        mant[0], E[0] = 1.0, -float(l)
        for i in range(1, n):  # the product itself: logarithms would lose digits
            mant[i], E[i] = mant[i - 1] * r[i], E[i - 1]
            if mant[i] > 1e100:
                mant[i], E[i] = mant[i] * 2.0 ** -300, E[i] + 300.0
        edge = torch.from_numpy(mant[::-1].copy()).to(DEV)
        ex = torch.from_numpy(E[::-1].copy()).to(DEV)
        sign = torch.where(((l - torch.arange(n, device=DEV)) & 1) == 1, -1.0, 1.0)
        self.cur[l, :n], self.E[l, :n], self.old[l, :n] = sign * edge, ex, 0.0
        self.cur[:n, l], self.E[:n, l], self.old[:n, l] = edge, ex, 0.0
        self.cur[l, l] = edge[l]
        e = self.E[:n, :n]
        half = torch.exp2(torch.clamp(e * 0.5, min=-1070.0))
        return self.cur[:n, :n] * half * half


def _angle(num, den):
    """pi * num / den with num reduced modulo 2 den (integers, exact)."""
    return (num % (2 * den)).double() * (math.pi / den)


class _Scale:
    """One field: kernel weights w[l] s_{l n_k}, its grid and its band."""

    def __init__(self, w, s, L, lg, band, mw):
        self.w, self.s, self.N, self.L, self.lg, self.band, self.mw = w, s, s.shape[1], L, lg, band, mw
        self.ns = [-(self.N - 1) + 2 * k for k in range(self.N)]
        self.nb, self.n = (lg if mw else 2 * lg), 2 * lg - 1
        self.G = None

    def beta(self):
        b = 2 * torch.arange(self.nb, device=DEV) + 1
        return b, (2 * self.lg - 1 if self.mw else 4 * self.lg)  # beta = pi b / den

    def trig(self):
        """cos and sin of m' beta_b, [nb][band]."""
        b, den = self.beta()
        a = _angle(b[:, None] * torch.arange(self.band, device=DEV), den)
        return torch.cos(a), torch.sin(a)


def _fields(L, N, lam, J0, grid):
    kap, phi = _radial(L, lam, J0)
    s = _direction(L, N)
    bands, bphi = _bands(kap, phi)
    out = []
    for j in range(len(bands)):
        lg = max(1, bands[j]) if grid == "multires" else L
        out.append(_Scale(kap[j], s, L, lg, bands[j], grid == "mw"))
    lg = bphi if grid == "multires" else L
    out.append(_Scale(phi, np.ones((L, 1), dtype=np.complex128), L, lg, bphi, grid == "mw"))
    return out


def _orders(D, l, ns):
    """Delta^l_{m' n} for the orders ns, [m' <= l][k] (zero where |n| > l)."""
    sgn = torch.where(((l + torch.arange(l + 1, device=DEV)) & 1) == 1, -1.0, 1.0)
    cols = []
    for n in ns:
        if abs(n) > l:
            cols.append(torch.zeros(l + 1, device=DEV, dtype=torch.float64))
        else:
            cols.append(D[:, abs(n)] if n >= 0 else sgn * D[:, abs(n)])
    return torch.stack(cols, 1)


def _analyse(f, fields, L, slabs=None):
    """The samples of every field (a list of [N][nb][n]); slabs: Delta^l for every l, if at hand."""
    f = f.to(torch.complex128)
    for s in fields:
        s.G = torch.zeros(s.N, s.band, s.band, device=DEV, dtype=torch.complex128)  # [k][m'][m]
    wig = _Wigner(L) if slabs is None else None
    for l in range(L):
        D = slabs[l] if wig is None else wig.step()
        A = D * f[l * l + l:l * l + 2 * l + 1]
        for s in fields:
            if l < s.band and s.w[l] > 0:
                coef = torch.from_numpy(s.w[l] * np.conj(s.s[l])).to(DEV)
                s.G[:, :l + 1, :l + 1] += A * (_orders(D, l, s.ns) * coef).T[:, :, None]
    out = []
    for s in fields:
        W = torch.zeros(s.N, s.nb, s.n, device=DEV, dtype=torch.float64)
        if s.band > 0:
            cb, sb = s.trig()
            m = torch.arange(s.band, device=DEV)
            X = []
            for k, n in enumerate(s.ns):
                U = s.G[k] * (1j ** ((n - m) % 4).to(torch.complex128))
                ev = ((m + n) % 2 == 0)
                two = torch.full((s.band, 1), 2.0, device=DEV, dtype=torch.float64)
                two[0] = 1.0
                U2 = U * two
                C = torch.complex(cb @ U2.real.contiguous(), cb @ U2.imag.contiguous())
                S = torch.complex(sb @ U2.real.contiguous(), sb @ U2.imag.contiguous())
                odd0 = torch.complex(torch.zeros((), device=DEV, dtype=torch.float64), torch.ones((), device=DEV, dtype=torch.float64))
                # m' = 0 enters once: cos(0) = 1 (even); its odd partner Delta_{0m} Delta_{0n} vanishes
                X.append(torch.where(ev[None, :], C, odd0 * S))
            X = torch.stack(X)  # [k][b][m]
            for g in range(s.N):
                ph = torch.tensor([complex(math.cos(math.pi * n * g / s.N), math.sin(math.pi * n * g / s.N))
                                   for n in s.ns], device=DEV, dtype=torch.complex128)
                Z = (X * ph[:, None, None]).sum(0)
                Z = torch.nn.functional.pad(torch.view_as_real(Z), (0, 0, 0, s.lg - s.band))
                W[g] = torch.fft.irfft(torch.view_as_complex(Z.contiguous()), n=s.n, norm="forward")
        s.G = None
        out.append(W)
    return out


def _dh_weights(L):
    t = 2 * torch.arange(2 * L, device=DEV) + 1
    k = 2 * torch.arange(L, device=DEV) + 1
    s = torch.sin(_angle(t[:, None] * k, 4 * L)) / k
    return 2.0 / L * torch.sin(_angle(t, 4 * L)) * s.sum(1)


def _synthesise(Ws, fields, L):
    """f_lm (m >= 0 and by symmetry m < 0) from samples on the DH grid."""
    for s, W in zip(fields, Ws):
        s.G = None
        if s.band == 0:
            continue
        cb, sb = s.trig()
        q = _dh_weights(s.lg)
        m = torch.arange(s.band, device=DEV)
        H = torch.zeros(s.N, s.band, s.band, device=DEV, dtype=torch.complex128)
        for g in range(s.N):
            V = torch.fft.rfft(W[g].double(), n=s.n)[:, :s.band] * (2.0 * math.pi / s.n)
            V = V * q[:, None]
            C = torch.complex(cb.T @ V.real.contiguous(), cb.T @ V.imag.contiguous())
            S = torch.complex(sb.T @ V.real.contiguous(), sb.T @ V.imag.contiguous())
            for k, n in enumerate(s.ns):
                x = -math.pi * n * g / s.N
                ph = complex(math.cos(x), math.sin(x)) * (2.0 * math.pi / s.N)
                T = torch.where(((m + n) % 2 == 0)[None, :], 2.0 * C, -2j * S)
                T[0] = torch.where((m + n) % 2 == 0, C[0], torch.zeros_like(C[0]))
                H[k] += ph * T
        for k, n in enumerate(s.ns):
            H[k] *= (1j ** ((m - n) % 4).to(torch.complex128))
        s.G = H
    out = torch.zeros(L * L, device=DEV, dtype=torch.complex128)
    wig = _Wigner(L)
    for l in range(L):
        D = wig.step()
        acc = torch.zeros(l + 1, device=DEV, dtype=torch.complex128)
        for i, s in enumerate(fields):
            if s.G is not None and l < s.band and s.w[l] > 0:
                norm = (2 * l + 1) / (4.0 * math.pi if i == len(fields) - 1 else 8.0 * math.pi ** 2)
                norm /= 2.0 * math.pi if i == len(fields) - 1 else 1.0  # its single gamma sample carries 2 pi
                coef = torch.from_numpy(s.w[l] * s.s[l]).to(DEV) * norm
                R = _orders(D, l, s.ns) * coef
                acc += (D * (R.T[:, :, None] * s.G[:, :l + 1, :l + 1]).sum(0)).sum(0)
        out[l * l + l:l * l + 2 * l + 1] = acc
        sgn = torch.where((torch.arange(1, l + 1, device=DEV) & 1) == 1, -1.0, 1.0)
        out[l * l:l * l + l] = (sgn * acc[1:].conj()).flip(0)
    for s in fields:
        s.G = None
    return out


def _join(case, Ws):
    W = Ws[:-1]
    return (torch.cat([w.reshape(-1) for w in W]) if case["grid"] == "multires" else torch.stack(W)), Ws[-1][0]


def exact(case, seed):
    L, N, op = case["L"], case["N"], case["op"]
    cd, rd = _dtypes(case)
    gen = _gen(seed)
    if op == "batch":
        Wb, Pb, gb = [], [], []
        fields = {}
        wig = _Wigner(case["L"])
        slabs = [wig.step() for _ in range(case["L"])]
        for a, b in _batch_config(case):
            f = _signal(a, gen, cd)
            if (a, b) not in fields:
                fields[(a, b)] = _fields(a, b, case["lam"], case["J0"], "dh")
            Ws = _analyse(f, fields[(a, b)], a, slabs)
            for dst, v in ((gb, f.to(torch.complex128)), (Wb, torch.stack(Ws[:-1]).reshape(-1)), (Pb, Ws[-1].reshape(-1))):
                dst.append(torch.cat([v, v.new_zeros(_up(v.numel()) - v.numel())]))
        return torch.cat(Wb), torch.cat(Pb), torch.cat(gb)
    if op == "sht":
        f = _signal(L, gen, cd)
        y = np.sqrt((2.0 * np.arange(L) + 1.0) / (4.0 * math.pi))
        field = _Scale(y, np.ones((L, 1), dtype=np.complex128), L, L, L, False)
        return _analyse(f, [field], L)[0][0], f.to(torch.complex128)
    fields = _fields(L, N, case["lam"], case["J0"], case["grid"])
    if op == "synthesis":
        shape = (len(fields) - 1, N, fields[0].nb, fields[0].n)
        W = torch.randn(shape, generator=gen, device=DEV, dtype=rd)
        Wphi = torch.randn(shape[2:], generator=gen, device=DEV, dtype=rd)
        return _synthesise(list(W) + [Wphi[None]], fields, L)
    f = _signal(L, gen, cd)
    got = _join(case, _analyse(f, fields, L))
    # the pair is exact for a band-limited real signal
    return got if op == "analysis" else got + (f.to(torch.complex128),)
