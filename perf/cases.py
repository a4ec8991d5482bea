"""The work a user of this framework has it do, as measurable cases.

Every case is one call of the public binding (``paper_2311_17174_gb300.emri``)
on seeded synthetic inputs of the recipes in ``inputs.py``:

* ``lnl``       emri_loglike_batch, or emri_loglike_batch_fd with ``fd``
* ``chains``    emri_loglike_multi (several chains in one graph)
* ``stretch``   emri_stretch_step (one ensemble step)
* ``waveform``  emri_ak_waveform
* ``fft``       emri_fft_batch

``listed()`` holds the sizes of the repository's own configurations;
``draw()`` spreads over the same ranges.  ``exact()`` restates the path in
plain numpy and torch (64-bit, the orbit in long double), sharing no code with
the library.
"""
from __future__ import annotations

import decimal
import math

import numpy as np
import torch

from paper_2311_17174_gb300 import emri
from paper_2311_17174_gb300 import inputs as I

DT = I.DT
FMIN, FMAX = 1e-4, 1.0
SNR = 50.0
F_STAR = 1e-2                     # pivot frequency of the propagation model
FD_MODEL = (2, 1)                 # alpha_M and alpha_T terms of the fd cases
STRETCH_FREE = (I.I_M, I.I_MU, I.I_SPIN, I.I_XI0)   # the paper's free parameters
#: walkers x samples above which exact() would take too long
EXACT_MOST = 1 << 25


# ------------------------------------------------------------------- cases
def listed():
    return [
        # the smallest request of the serving mix: launches and latency count
        {"name": "lnl mixed 8w 2^16", "do": "lnl", "w": 8, "logn": 16, "n_max": 10, "mixed": True, "src": "scatter"},
        # 16 independent sources, 2^16 samples, n <= 10, FP64 (catalogue pass)
        {"name": "lnl fp64 16src 2^16", "do": "lnl", "w": 16, "logn": 16, "n_max": 10, "mixed": False,
         "src": "sources"},
        # the paper's own workload: 8 walkers, one year, backward from the LSO
        {"name": "lnl fp64 paper 8w", "do": "lnl", "w": 8, "logn": 21, "n_max": 10, "mixed": False, "src": "paper"},
        {"name": "lnl mixed paper 8w", "do": "lnl", "w": 8, "logn": 21, "n_max": 10, "mixed": True, "src": "paper"},
        # one GPU's block (128 walkers) of the 1024-walker ensemble, FP64
        {"name": "lnl fp64 128w 2^21", "do": "lnl", "w": 128, "logn": 21, "n_max": 20, "mixed": False,
         "src": "scatter"},
        # the whole 1024-walker ensemble, one year, mixed precision
        {"name": "lnl mixed 1024w 2^21", "do": "lnl", "w": 1024, "logn": 21, "n_max": 20, "mixed": True,
         "src": "scatter"},
        # frequency-dependent propagation, an odd walker count
        {"name": "lnl fd mixed 333w 2^18", "do": "lnl", "w": 333, "logn": 18, "n_max": 15, "mixed": True,
         "src": "scatter", "fd": True},
        # uneven chains (32..512 walkers, 2^16..2^20 samples, n 5..30), one graph
        {"name": "chains mixed 8", "do": "chains", "chains": 8, "w_lo": 32, "w_hi": 512, "log_lo": 16, "log_hi": 20,
         "mixed": True},
        # one ensemble step of the sampler, FP64, an odd half size
        {"name": "stretch fp64 98w 2^18", "do": "stretch", "w": 98, "logn": 18, "n_max": 20},
        # the time series themselves: a handful of sources
        {"name": "waveform fp64 5src 2^20", "do": "waveform", "w": 5, "logn": 20, "n_max": 20, "mixed": False},
        # spectra of stored series, forward FP64 and inverse FP32 (odd batches)
        {"name": "fft fp64 forward 23x2^19", "do": "fft", "batch": 23, "logn": 19, "mixed": False, "sign": -1},
        {"name": "fft fp32 inverse 75x2^20", "do": "fft", "batch": 75, "logn": 20, "mixed": True, "sign": 1},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    do = rng.choice(["lnl", "lnl", "lnl", "waveform", "fft", "stretch", "chains"])
    mixed = rng.random() < 0.5
    logn = rng.randint(16, 21)
    n = 1 << logn
    most = (1 << 28) if mixed else (1 << 25)        # walkers x samples of one pass
    w = _log_int(rng, 1, max(2, min(512, most // n)))
    n_max = rng.randint(5, 30)
    if do == "lnl":
        return {"do": do, "w": w, "logn": logn, "n_max": n_max, "mixed": mixed,
                "src": rng.choice(["scatter", "sources", "paper"]), "fd": rng.random() < 0.25}
    if do == "waveform":
        return {"do": do, "w": _log_int(rng, 1, max(2, min(64, (1 << 24) // n))), "logn": logn, "n_max": n_max,
                "mixed": mixed}
    if do == "fft":
        logn = rng.randint(12, 21)
        return {"do": do, "batch": _log_int(rng, 1, max(2, (1 << 25) >> logn)), "logn": logn, "mixed": mixed,
                "sign": rng.choice([-1, 1])}
    if do == "stretch":
        logn = rng.randint(16, 18)
        return {"do": do, "w": 2 * _log_int(rng, 4, 64) + rng.randint(0, 1), "logn": logn, "n_max": n_max}
    lo = rng.randint(16, 18)
    return {"do": "chains", "chains": rng.randint(2, 8), "w_lo": 8, "w_hi": rng.randint(32, 128), "log_lo": lo,
            "log_hi": lo + rng.randint(0, 1), "mixed": mixed}


def _chain_list(case, seed):
    """(walkers, log2 n, n_max) of each chain: the sizes are the case's, the same for every seed."""
    g = np.random.default_rng([case["chains"], case["w_hi"], case["log_lo"]])
    return [(int(g.integers(case["w_lo"], case["w_hi"] + 1)), int(g.integers(case["log_lo"], case["log_hi"] + 1)),
             int(g.integers(5, 31))) for _ in range(case["chains"])]


def work(case):
    """Each input read once, each output written once; flops of the factored
    harmonic sum (24 per harmonic, 172 for phases, response and channels), the
    FFT (5 log2 n) and the inner products (20 per bin)."""
    if case["do"] == "fft":
        n, cs = 1 << case["logn"], 8 if case["mixed"] else 16
        return {"bytes": 2.0 * case["batch"] * n * cs, "flops": 5.0 * case["batch"] * n * case["logn"]}
    if case["do"] == "chains":
        parts = _chain_list(case, 0)
    else:
        parts = [(case["w"], case["logn"], case["n_max"])]
    mixed = case.get("mixed", False)
    bytes_, flops = 0.0, 0.0
    for w, logn, n_max in parts:
        n = 1 << logn
        bytes_ += w * (16 * 8 + 28)
        flops += float(w) * n * (24 * n_max + 172)
        if case["do"] == "waveform":
            bytes_ += float(w) * n * (8 if mixed else 16)
        else:
            bytes_ += n * (12 if mixed else 24)
            flops += float(w) * n * (5 * logn + 20)
    return {"bytes": bytes_, "flops": flops}


# ------------------------------------------------------------------ inputs
def _dev(a):
    return torch.as_tensor(np.ascontiguousarray(a, dtype=np.float64)).to(_device())


def _device():
    return torch.device("cuda:0" if torch.cuda.is_available() else "cpu")


def _problem(seed, src, w, logn, n_max, fd=False):
    """Walkers, data and noise curve of one dataset: an injection at SNR 50
    (noise-free at 1 Gpc for the paper's workload), its spectrum plus seeded
    noise, and the walkers scattered about it (or independent sources)."""
    n = 1 << logn
    psd = I.psd_bc04(n, DT)
    back = src == "paper"
    if back:
        wl = I.config_paper(walkers=w, n=n, n_max=n_max, seed=seed)
        th, inj = wl.theta, wl.injection
    else:
        th = I.draw_sources(seed, w if src == "sources" else 1, n)
        inj = th[0].copy()
    spec = torch.fft.fft(_waveform(inj[None], n, n_max, back, np.float64)[0])
    wk = _weights(psd, n)
    hh = float((wk * (spec.real ** 2 + spec.imag ** 2)).sum())
    target = 1e3 * _MPC if back else math.sqrt(hh) / SNR
    z = I.solve_distance(target, lambda zz: _distance(zz) * float(_xi(zz, inj[I.I_XI0])))
    inj[I.I_Z] = z
    th[:, I.I_Z] = z if back else th[:, I.I_Z]
    if src != "paper":
        if src == "scatter":
            th = I.scatter_walkers(seed + 1, inj, w)
        else:
            th[0] = inj
    data = spec * _delay(inj, n) / (_distance(z) * float(_xi(z, inj[I.I_XI0])))
    if not back:
        data = data + torch.as_tensor(I.noise_spectrum(seed + 2, psd, n, DT)).to(data.device)
    coef = None
    if fd:
        coef = np.random.default_rng(seed + 3).normal(0.0, 0.05, (sum(FD_MODEL), w))
    return {"theta": th, "n": n, "n_max": n_max, "psd": psd, "data": data, "coef": coef, "back": back}


def _opts(p, mixed):
    return emri.opts(precision=emri.MIXED if mixed else emri.FP64, n_max=p["n_max"],
                     mode=emri.BACKWARD_FROM_LSO if p["back"] else emri.FORWARD)


def _problems(case, seed):
    if case["do"] == "chains":
        return [_problem(seed * 64 + i, "scatter", w, logn, n_max)
                for i, (w, logn, n_max) in enumerate(_chain_list(case, seed))]
    return [_problem(seed * 64, case.get("src", "scatter"), case["w"], case["logn"], case["n_max"],
                     case.get("fd", False))]


def _fft_input(case, seed):
    """Packed two-channel series: noise-like samples, as stored strain is."""
    g = torch.Generator(device=_device()).manual_seed(seed)
    real = torch.float32 if case["mixed"] else torch.float64
    x = torch.randn((case["batch"], 1 << case["logn"], 2), generator=g, device=_device(), dtype=real)
    return torch.view_as_complex(x)


def _uniforms(case, seed):
    return np.random.default_rng(seed * 64 + 5).random((3, case["w"]))


def _box(inj):
    return [float(v) - abs(float(v)) for v in inj], [float(v) + abs(float(v)) for v in inj]


def prepare(case, seed):
    ctx = emri.Context(0)
    s = {"do": case["do"], "ctx": ctx}
    if case["do"] == "fft":
        s["src"] = _fft_input(case, seed)
        s["z"] = torch.empty_like(s["src"])
        s["args"] = (1 << case["logn"], case["batch"], emri.MIXED if case["mixed"] else emri.FP64, case["sign"])
        return s
    mixed = case.get("mixed", False)
    if case["do"] == "waveform":
        n = 1 << case["logn"]
        s["grid"] = emri.grid(n, DT)
        s["theta"] = _dev(I.draw_sources(seed * 64, case["w"], n).T)
        s["opts"] = emri.opts(precision=emri.MIXED if mixed else emri.FP64, n_max=case["n_max"])
        s["z"] = torch.empty((case["w"], n), dtype=torch.complex64 if mixed else torch.complex128, device="cuda:0")
        s["status"] = torch.empty(case["w"], dtype=torch.int32, device="cuda:0")
        return s
    s["items"], s["mixed"] = [], mixed
    for p in _problems(case, seed):
        w = p["theta"].shape[0]
        ds = ctx.dataset(emri.grid(p["n"], DT), p["data"], p["psd"], FMIN, FMAX)
        out = [torch.empty(w, dtype=torch.float64, device="cuda:0") for _ in range(3)]
        status = torch.empty(w, dtype=torch.int32, device="cuda:0")
        # in mixed precision a sampler asks for lnL and the status words only
        dh_hh = [None, None] if mixed else out[1:]
        s["items"].append((ds, _dev(p["theta"].T), _opts(p, mixed), out[0], *dh_hh, status))
    if case.get("fd"):
        s["coef"] = _dev(p["coef"])
    if case["do"] == "stretch":
        lo, hi = _box(p["theta"][0])
        s["cfg"] = emri.stretch_cfg(STRETCH_FREE, lo, hi)
        s["u"] = _dev(_uniforms(case, seed))
        s["accepted"] = torch.empty(case["w"], dtype=torch.int32, device="cuda:0")
        ctx.loglike_batch(*s["items"][0])            # lnP of the starting ensemble
    return s


def run(s):
    ctx = s["ctx"]
    if s["do"] == "fft":
        s["z"].copy_(s["src"])                       # the transform is in place; the series is kept
        ctx.fft_batch(s["z"], *s["args"])
        return s["z"]
    if s["do"] == "waveform":
        ctx.ak_waveform(s["grid"], s["theta"], s["opts"], s["z"], s["status"])
        return {"z": s["z"], "status": s["status"]}
    if s["do"] == "stretch":
        ds, theta, o, lnl = s["items"][0][:4]
        ctx.stretch_step(ds, theta, lnl, o, s["cfg"], s["u"], s["accepted"])
        return {"theta": theta, "lnp": lnl, "accepted": s["accepted"]}
    if s["do"] == "chains":
        ctx.loglike_multi(s["items"])
    elif "coef" in s:
        ds, theta, o, *out = s["items"][0]
        ctx.loglike_batch_fd(ds, theta, o, *FD_MODEL, F_STAR, s["coef"], *out)
    else:
        ctx.loglike_batch(*s["items"][0])
    res = []
    for _, _, _, lnl, dh, hh, status in s["items"]:
        # the mixed path sums in FP32: its log-likelihoods are kept in that type
        res.append({"lnl": lnl.float() if s["mixed"] else lnl, "status": status} if dh is None else
                   {"lnl": lnl, "dh": dh, "hh": hh, "status": status})
    return res


# ------------------------------------------------------ the path, restated
_GMSUN, _C, _MPC = 1.32712440018e26, 2.99792458e10, 3.0856775814913673e24   # cgs
_AU_C, _YEAR = 499.004783836, 31557600.0                                      # [s]
_OM, _H0 = 0.315, 67.4
_M = 32                                                                       # nodes per segment
_SEG = 16384                                                                  # samples per segment


def _xi(z, xi0):
    return xi0 + (1.0 - xi0) / (1.0 + z) ** 2


def _distance(z):
    """Luminosity distance [cm], flat Lambda-CDM."""
    x, w = np.polynomial.legendre.leggauss(48)
    a = 1.0 + 0.5 * z * (x + 1.0)
    return (1.0 + z) * _C * _MPC / (_H0 * 1e5) * 0.5 * z * float(np.sum(w / np.sqrt(_OM * a ** 3 + 1.0 - _OM)))


def _weights(psd, n):
    """w_k = 2 dt^2 df / S in the band, without DC and Nyquist."""
    df = 1.0 / (n * DT)
    k = np.arange(n)
    k = np.minimum(k, n - k)
    f = k * df
    ok = (k > 0) & (2 * k < n) & (f >= FMIN) & (f <= FMAX)
    return torch.as_tensor(np.where(ok, 2.0 * DT * DT * df / psd[k], 0.0)).to(_device())


def _lookback(z):
    """t_LB [s] to 60 digits."""
    D = decimal.Decimal
    om = D(_OM)
    s = ((1 - om) / om).sqrt()
    zp = 1 + D(float(z))
    u = s / (zp * zp.sqrt())
    asinh = lambda a: (a + (a * a + 1).sqrt()).ln()  # noqa: E731
    return D(_MPC) / (D(_H0) * D(10) ** 5) * 2 / (3 * (1 - om).sqrt()) * (asinh(s) - asinh(u))


def _phase_mod1(fracs, powers, k):
    """sum_m fracs[m] 2^-128 k^powers[m] mod 1 (k integers >= 0) in 128-bit fixed point: four
    32-bit limbs in uint64."""
    mask = np.uint64(0xFFFFFFFF)
    kk = k.astype(np.uint64)
    tot = [np.zeros_like(kk) for _ in range(4)]
    for v, p in zip(fracs, powers):
        limbs = [np.full_like(kk, (v >> (32 * i)) & 0xFFFFFFFF) for i in range(4)]
        for _ in range(p):
            carry = np.zeros_like(kk)
            for i in range(4):
                t = limbs[i] * kk + carry
                limbs[i], carry = t & mask, t >> np.uint64(32)
        carry = np.zeros_like(kk)
        for i in range(4):
            t = tot[i] + limbs[i] + carry
            tot[i], carry = t & mask, t >> np.uint64(32)
    return tot[3].astype(np.float64) / 2.0 ** 32 + tot[2].astype(np.float64) / 2.0 ** 64


def _delay(th, n, b=(), f_star=F_STAR):
    """exp(-2 pi i k_s frac(dt_GW / T)) over the bins, with the frequency-dependent terms b."""
    with decimal.localcontext() as cx:
        cx.prec = 80
        D = decimal.Decimal
        t = D(n) * D(DT)
        half = -_lookback(th[I.I_Z]) / 2
        terms = [D(float(th[I.I_ALPT])) * half / t]
        terms += [D(float(v)) * half / t / (t * D(f_star)) ** (m + 1) for m, v in enumerate(b)]
        ints = [int(v * (1 << 128)) % (1 << 128) for v in terms]
    k = np.arange(n)
    a = np.where(2 * k <= n, k, n - k)
    neg = 2 * k > n
    ph = _phase_mod1(ints, range(1, len(ints) + 1), a)
    # the Nyquist bin carries no weight; its sign does not matter
    ph = torch.as_tensor(np.where(neg, -ph, ph)).to(_device()) * (-2.0 * math.pi)
    return torch.polar(torch.ones_like(ph), ph)


def _cheb_tables(x, real):
    """Values and integrals (over the unit segment) at x in [-1, 1] of the
    Lagrange basis at the Chebyshev-Lobatto nodes."""
    m = _M
    j = np.arange(m).astype(real)
    nodes = -np.cos(np.arccos(real(-1)) * j / (m - 1))
    c = np.ones(m, real)
    c[0] = c[-1] = 2

    def cheb(y, top):
        t = [np.ones_like(y), y]
        for _ in range(2, top):
            t.append(2 * y * t[-1] - t[-2])
        return np.stack(t)

    tn = cheb(nodes, m)                                            # [k, j]
    coef = 2 / ((m - 1) * c[:, None] * c[None, :]) * tn            # [k, j]: nodal values -> Chebyshev
    tx = cheb(x.astype(real), m + 1)
    ends = cheb(np.array([-1.0]).astype(real), m + 1)

    def prim(t):
        out = [t[1], t[2] / 4]
        for k in range(2, m):
            out.append(t[k + 1] / (2 * (k + 1)) - t[k - 1] / (2 * (k - 1)))
        return np.stack(out)

    integ = (prim(tx) - prim(ends)) / 2
    return (coef.T @ tx[:m]).T, (coef.T @ integ).T                 # [x, j] each


def _rates(c, v, e):
    """AK right-hand side in v = (2 pi M nu)^(1/3); angles in cycles."""
    e2 = e * e
    e4, om = e2 * e2, 1 - e2
    e6 = e4 * e2
    s = 1 / np.sqrt(om)
    s2 = s * s
    s3 = s2 * s
    v2 = v * v
    v3 = v2 * v
    v8 = v2 * v2 * v2 * v2
    one = c["one"]
    aS, cl = c["spin"], c["cl"]
    br = (1 + 73 * one / 24 * e2 + 37 * one / 96 * e4) * om
    br = br + v2 * (1273 * one / 336 - 2561 * one / 224 * e2 - 3885 * one / 128 * e4 - 13147 * one / 5376 * e6)
    br = br - v3 * aS * cl * s * (73 * one / 12 + 1211 * one / 24 * e2 + 3143 * one / 96 * e4 + 65 * one / 64 * e6)
    eb = (304 + 121 * e2) * om * (1 + 12 * v2) - v2 / 56 * (8 * 16705 + 12 * 9082 * e2 - 25211 * e4)
    s7 = s3 * s3 * s
    dv = c["kv"] * v8 * v * s7 * s2 * br
    de = -e / 15 * c["ke"] * s7 * v8 * eb
    de = de + e * c["ke"] * aS * cl * v8 * v3 * s7 * s * (1364 * one / 5 + 5032 * one / 15 * e2 + 263 * one / 10 * e4)
    nu = v3 * c["inv"]
    g = 3 * nu * v2 * s2 * (1 + v2 * s2 * (26 - 15 * e2) / 4) - 6 * nu * cl * aS * v3 * s3
    return dv, de, nu, g, 2 * nu * aS * v3 * s3


def _orbit(th, n, back, real):
    """Per segment: the state at its first sample and the five rates at its
    Chebyshev nodes ([W, segments, 32]), in `real`."""
    w = th.shape[0]
    seg = min(n, _SEG)
    one = real(1)
    tsun = real(_GMSUN) / (real(_C) ** 3)
    m, mu = th[:, I.I_M].astype(real) * tsun, th[:, I.I_MU].astype(real) * tsun
    col = lambda a: a[:, None]  # noqa: E731
    pi = np.arccos(real(-1))
    c = {"one": one, "spin": col(th[:, I.I_SPIN].astype(real)), "cl": col(np.cos(th[:, I.I_LAM].astype(real))),
         "kv": col(32 * mu / (5 * m * m)), "ke": col(mu / (m * m)), "inv": col(1 / (2 * pi * m))}
    e0 = th[:, I.I_E0].astype(real)
    if back:
        x0 = ((1 - e0 * e0) / (6 + 2 * e0)) ** (one * 3 / 2)
    else:
        x0 = 2 * pi * m * th[:, I.I_NU0].astype(real)
    y = [col(np.cbrt(x0)), col(e0)]
    y += [col(th[:, q].astype(real) / (2 * pi)) for q in (I.I_PHI0, I.I_GAM0, I.I_ALP0)]
    _, qn = _cheb_tables(-np.cos(np.pi * np.arange(_M).astype(real) / (_M - 1)), real)
    qnt = qn.T.copy()
    if back:        # the start state sits at the last sample: one RK4 step to sample n
        h = real(DT)
        k1 = _rates(c, y[0], y[1])
        k2 = _rates(c, y[0] + h / 2 * k1[0], y[1] + h / 2 * k1[1])
        k3 = _rates(c, y[0] + h / 2 * k2[0], y[1] + h / 2 * k2[1])
        k4 = _rates(c, y[0] + h * k3[0], y[1] + h * k3[1])
        y = [y[q] + h / 6 * (k1[q] + 2 * k2[q] + 2 * k3[q] + k4[q]) for q in range(5)]
    hseg = real(DT) * seg * (-1 if back else 1)
    tol = 1e-18 if real is np.longdouble else 1e-15
    nseg = n // seg
    start, nodes = [None] * nseg, [None] * nseg
    for g in (range(nseg - 1, -1, -1) if back else range(nseg)):
        v, e = y[0] + np.zeros((w, _M), real), y[1] + np.zeros((w, _M), real)
        for _ in range(40):
            f = _rates(c, v, e)
            vn, en = y[0] + hseg * (f[0] @ qnt), y[1] + hseg * (f[1] @ qnt)
            done = np.max(np.abs(vn - v)) < tol and np.max(np.abs(en - e)) < tol
            v, e = vn, en
            if done:
                break
        f = _rates(c, v, e)
        end = [y[q] + hseg * (f[q] @ qnt[:, -1:]) for q in range(5)]
        first, f = (end, [r[:, ::-1] for r in f]) if back else (y, f)
        for q in (2, 3, 4):
            end[q] = end[q] - np.floor(end[q])
        start[g] = np.stack([a[:, 0] for a in first], -1)
        nodes[g] = np.stack(f, -1)
        y = end
    return np.stack(start, 1), np.stack(nodes, 1), m, mu              # [W, G, 5], [W, G, 32, 5]


def _bessel(x, top):
    """J_0..J_top(x), by downward recurrence normalised with J_0 + 2 sum J_2k = 1."""
    m = 2 * ((max(top, int(np.max(x))) + 40) // 2)
    x = np.maximum(x, 1e-300)
    hi, lo = np.zeros_like(x), np.full_like(x, 1e-280)
    out, norm = {}, np.zeros_like(x)
    for k in range(m, 0, -1):
        cur = 2 * k / x * lo - hi
        hi, lo = lo, cur
        big = np.abs(lo) > 1e200
        if big.any():
            s = np.where(big, 1e-200, 1.0)
            hi, lo, norm = hi * s, lo * s, norm * s
            out = {q: a * s for q, a in out.items()}
        if k - 1 <= top:
            out[k - 1] = lo
        if (k - 1) % 2 == 0:
            norm = norm + (lo if k == 1 else 2 * lo)
    return [out[q] / norm for q in range(top + 1)]


def _amplitudes(e, n_max):
    """n pa, n sqrt(1-e^2) pb, 2 pc of every harmonic at eccentricities e."""
    res = []
    for n in range(1, n_max + 1):
        j = _bessel(n * e, n + 2)
        jm2 = -j[1] if n == 1 else j[n - 2]
        a = jm2 - 2 * e * j[n - 1] + 2 / n * j[n] + 2 * e * j[n + 1] - j[n + 2]
        b = np.sqrt(1 - e * e) * (jm2 - 2 * j[n] + j[n + 2])
        res += [n * a, n * b, 2 * j[n]]
    return np.stack(res, -1)                                         # [..., 3 n_max]


def _waveform(th, n, n_max, back, real=np.longdouble):
    """[W, n] complex128: h_I + i h_II at unit distance."""
    dev = _device()
    seg = min(n, _SEG)
    start, rate, m, mu = _orbit(th, n, back, real)
    w, nseg = start.shape[:2]
    h = DT * seg
    tau = np.arange(seg) / seg
    val, integ = _cheb_tables(2 * tau - 1, np.float64)
    _, qn = _cheb_tables(-np.cos(np.pi * np.arange(_M) / (_M - 1)), np.float64)
    e_nodes = start[:, :, 1, None].astype(np.float64) + h * (rate[..., 1].astype(np.float64) @ qn.T)
    t64 = lambda a: torch.as_tensor(np.ascontiguousarray(np.asarray(a, dtype=np.float64))).to(dev)  # noqa: E731
    val, integ = t64(val), t64(integ)
    j = torch.arange(seg, device=dev, dtype=torch.float64)
    z = torch.zeros((w, n), dtype=torch.complex128, device=dev)
    per = max(1, min(nseg, (1 << 18) // seg))                        # segments at a time
    for k in range(w):
        amp_nodes = t64(_amplitudes(e_nodes[k], n_max))
        ths, phs, thk, phk, lam = (float(th[k, q]) for q in (I.I_THS, I.I_PHS, I.I_THK, I.I_PHK, I.I_LAM))
        big_n = np.array([math.sin(ths) * math.cos(phs), math.sin(ths) * math.sin(phs), math.cos(ths)])
        spin = np.array([math.sin(thk) * math.cos(phk), math.sin(thk) * math.sin(phk), math.cos(thk)])
        e1 = (np.array([0.0, 0.0, 1.0]) - spin * math.cos(thk)) / math.sin(thk)
        e2 = np.cross(spin, e1)
        pol_p = np.array([-math.sin(phs), math.cos(phs), 0.0])
        pol_q = np.cross(pol_p, big_n)
        inv = 1.0 / (2.0 * math.pi * float(m[k]))
        for g0 in range(0, nseg, per):
            gs = slice(g0, min(nseg, g0 + per))
            r0 = rate[k, gs, :1, :]
            dev_r = t64(rate[k, gs] - r0)                            # rates less the first node's
            inc = r0[:, 0, :] * real(DT)                             # per sample, split for exact products
            hi = np.round(np.asarray(inc * real(2 ** 30), np.float64)) / 2.0 ** 30
            lo = np.asarray(inc - hi.astype(real), np.float64)
            base = np.asarray(start[k, gs], np.float64)
            corr = h * torch.einsum("sj,gjq->gsq", integ, dev_r)

            def state(q):
                a = j * t64(hi[:, q])[:, None]
                if q >= 2:
                    a = a - torch.floor(a)
                return (a + j * t64(lo[:, q])[:, None] + corr[..., q] + t64(base[:, q])[:, None]).reshape(-1)

            v, e = state(0), state(1)
            t = (torch.arange(v.numel(), device=dev, dtype=torch.float64) + g0 * seg) * DT
            pb = 2.0 * math.pi * (t / _YEAR)
            cb, sb = torch.cos(pb), torch.sin(pb)
            cdp, sdp = cb * math.cos(phs) + sb * math.sin(phs), sb * math.cos(phs) - cb * math.sin(phs)
            phi = 2 * math.pi * torch.frac(state(2) + v ** 3 * inv * (_AU_C * math.sin(ths)) * cdp)
            gam2, alp = 4 * math.pi * torch.frac(state(3)), 2 * math.pi * torch.frac(state(4))
            amp = torch.einsum("sj,gja->gsa", val, amp_nodes[gs]).reshape(-1, 3 * n_max)
            cs = torch.zeros_like(phi)
            ss, rs = torch.zeros_like(phi), torch.zeros_like(phi)
            for q in range(1, n_max + 1):
                a, b, c = amp[:, 3 * q - 3], amp[:, 3 * q - 2], amp[:, 3 * q - 1]
                cq, sq = torch.cos(q * phi), torch.sin(q * phi)
                cs += a * cq
                ss += b * sq
                rs += c * cq
            # quadrupole in the orbital plane, projected on the sky basis (P, Q)
            ca, sa = torch.cos(alp), torch.sin(alp)
            u1 = [sa * e1[i] - ca * e2[i] for i in range(3)]
            u2 = [math.cos(lam) * (ca * e1[i] + sa * e2[i]) - math.sin(lam) * spin[i] for i in range(3)]
            dot = lambda a, b: sum(a[i] * float(b[i]) for i in range(3))  # noqa: E731
            x = cs * torch.cos(gam2) - ss * torch.sin(gam2)
            y = cs * torch.sin(gam2) + ss * torch.cos(gam2)
            p1, q1, p2, q2 = dot(u1, pol_p), dot(u1, pol_q), dot(u2, pol_p), dot(u2, pol_q)
            hp = (rs + x) * (p1 * p1 - q1 * q1) + (rs - x) * (p2 * p2 - q2 * q2) + 2 * y * (p1 * p2 - q1 * q2)
            hx = 2 * ((rs + x) * p1 * q1 + (rs - x) * p2 * q2 + y * (p1 * q2 + q1 * p2))
            # detector: normal z_d tilted 60 degrees towards the Sun, arms turning with phibar
            ct = 0.5 * math.cos(ths) - 0.75 ** 0.5 * math.sin(ths) * cdp
            az = pb + torch.atan2(3 ** 0.5 * math.cos(ths) + math.sin(ths) * cdp, 2 * math.sin(ths) * sdp)
            psi = torch.atan2(0.75 ** 0.5 * math.cos(ths) * cdp + 0.5 * math.sin(ths), 0.75 ** 0.5 * sdp)
            f1, f2 = 0.5 * (1 + ct * ct) * torch.cos(2 * psi), 0.5 * (1 + ct * ct) * torch.sin(2 * psi)
            g1, g2 = ct * torch.sin(2 * psi), ct * torch.cos(2 * psi)
            c2, s2 = torch.cos(2 * az), torch.sin(2 * az)
            h1 = (c2 * f1 - s2 * g1) * hp + (c2 * f2 + s2 * g2) * hx
            h2 = (s2 * f1 + c2 * g1) * hp + (s2 * f2 - c2 * g2) * hx
            scale = 0.75 ** 0.5 * v * v * (float(mu[k]) * _C)
            out = torch.complex(scale * h1, scale * h2)
            past = torch.zeros_like(v, dtype=torch.bool) if back else v * v >= (1 - e * e) / (6 + 2 * e)
            if bool(past.any()):                                     # zero from the plunge on
                out[int(torch.argmax(past.to(torch.int8))):] = 0
                z[k, g0 * seg: g0 * seg + out.numel()] = out
                break
            z[k, g0 * seg: g0 * seg + out.numel()] = out
    return z


def _exact_lnl(p, theta=None):
    """(lnl, dh, hh) of the problem's walkers (or of `theta` [W, 16])."""
    th = p["theta"] if theta is None else theta
    n = p["n"]
    wk = _weights(p["psd"], n)
    k = np.arange(n)
    a = torch.as_tensor(np.where(2 * k <= n, k, n - k).astype(np.float64)).to(_device())
    res = []
    for i in range(th.shape[0]):
        spec = torch.fft.fft(_waveform(th[i: i + 1], n, p["n_max"], p["back"])[0])
        z = float(th[i, I.I_Z])
        b = ()
        if p["coef"] is not None:
            qm = FD_MODEL[0]
            x = a / (n * DT * F_STAR)
            alpha_m = sum(float(p["coef"][q, i]) * x ** (q + 1) for q in range(qm))
            spec = spec * torch.exp(-0.5 * math.log1p(z) * alpha_m)
            b = [float(p["coef"][q, i]) for q in range(qm, sum(FD_MODEL))]
        hh = float((wk * (spec.real ** 2 + spec.imag ** 2)).sum())
        spec = spec * _delay(th[i], n, b)
        dh = float((wk * (p["data"].real * spec.real + p["data"].imag * spec.imag)).sum())
        d = _distance(z) * float(_xi(z, th[i, I.I_XI0]))
        res.append((dh / d - 0.5 * hh / (d * d), dh, hh))
    return np.array(res).T


def exact(case, seed):
    if case["do"] == "fft":
        x = _fft_input(case, seed).to(torch.complex128)
        z = torch.fft.fft(x) if case["sign"] < 0 else torch.fft.ifft(x) * float(1 << case["logn"])
        return z
    size = sum(w << logn for w, logn, _ in _chain_list(case, seed)) if case["do"] == "chains" \
        else case["w"] << case["logn"]
    if size > EXACT_MOST:
        return None
    if case["do"] == "waveform":
        n = 1 << case["logn"]
        return {"z": _waveform(I.draw_sources(seed * 64, case["w"], n), n, case["n_max"], False), "status": None}
    ps = _problems(case, seed)
    if case["do"] == "stretch":
        return _exact_step(case, seed, ps[0])
    res = []
    for p in ps:
        lnl, dh, hh = _exact_lnl(p)
        res.append({"lnl": lnl, "status": None} if case["mixed"] else {"lnl": lnl, "dh": dh, "hh": hh, "status": None})
    return res


def _exact_step(case, seed, p):
    """One stretch move (a = 2) of the two halves in turn."""
    th, w = p["theta"].copy(), case["w"]
    u = _uniforms(case, seed)
    lo, hi = _box(p["theta"][0])
    lnp = _exact_lnl(p)[0]
    half = w // 2
    free = list(STRETCH_FREE)
    for a0, a1, o0, o1 in ((0, half, half, w), (half, w, 0, half)):
        k = np.arange(a0, a1)
        j = o0 + np.minimum((u[0, k] * (o1 - o0)).astype(int), o1 - o0 - 1)
        t = u[1, k] + 1.0
        zz = t * t / 2.0
        y = th[k].copy()
        for q in free:
            y[:, q] = th[j, q] + zz * (th[k, q] - th[j, q])
        ly = _exact_lnl(p, y)[0]
        ok = np.all([(y[:, q] >= lo[q]) & (y[:, q] <= hi[q]) for q in free], axis=0)
        ok &= (len(free) - 1) * np.log(zz) + ly - lnp[k] - np.log(u[2, k]) > 0
        th[k[ok]], lnp[k[ok]] = y[ok], ly[ok]
    return {"theta": np.ascontiguousarray(th.T), "lnp": lnp, "accepted": None}
