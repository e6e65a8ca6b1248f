"""The library's performance cases: what a parameter-estimation program has it do, call by call.

A case names a public entry point (``kind``), its precision, detectors, observation time, batch size
and mode mask. ``prepare`` makes what the program holds before the call (data on the grid, detector
handles, parameter samples, and the plan, summary data or network where the entry point takes one),
``run`` makes one call, ``work`` counts what the call cannot do without, and ``exact`` evaluates the
same quantity in plain 64-bit torch.

Sizes are those of the repository's workloads (bins of [1e-4, 5e-2] Hz; LISA 2^22 s, Taiji 2^21 s,
TianQin 2^20 s; modes 22/21/33/32/44; batches of 1 to thousands) and the paper's 655360 s span.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2602_12011_gb300 import _lib as L
from paper_2602_12011_gb300 import workloads as W
from paper_2602_12011_gb300 import autograd as G

DEV = "cuda"
ALL = W.MODE_ALL
NETWORK = "LISA+Taiji+TianQin"
PREC = {"fp64": 0, "mixed": L.PE_PREC_MIXED}
HET_BINS = 256


def listed():
    return [
        # one point of a sampler that calls per sample from the host: (2,2), one detector, 2^20 s
        dict(name="single_22_host", kind="loglike", prec="fp64", dets="LISA", T=2.0 ** 20, B=1, mask=W.MODE_22, tdi=20, host=True),
        # one point with higher modes on the longest grid, parameters on the device
        dict(name="single_hm", kind="loglike", prec="fp64", dets="LISA", T=2.0 ** 22, B=1, mask=ALL, tdi=20, host=False),
        # an ensemble sampler's walkers on the three-detector network, through a plan refilled each step
        dict(name="walkers_network_plan", kind="plan", prec="fp64", dets=NETWORK, T=2.0 ** 22, B=45, mask=ALL, tdi=20, host=False),
        # the batched higher-mode likelihood over the prior (nested sampling's live points)
        dict(name="batch_hm", kind="loglike", prec="fp64", dets="LISA", T=2.0 ** 22, B=1024, mask=ALL, tdi=20, host=False),
        # the same batch at the mixed precision
        dict(name="batch_hm_mixed", kind="loglike", prec="mixed", dets="LISA", T=2.0 ** 22, B=1024, mask=ALL, tdi=20, host=False),
        # an odd batch on the network at the mixed precision
        dict(name="network_mixed", kind="loglike", prec="mixed", dets=NETWORK, T=2.0 ** 22, B=601, mask=ALL, tdi=20, host=False),
        # gradients of a set of Hamiltonian Monte Carlo chains (forward and backward)
        dict(name="grad_hm", kind="grad", prec="fp64", dets="LISA", T=2.0 ** 22, B=64, mask=ALL, tdi=20, host=False),
        # gradients of a large batch at the mixed precision
        dict(name="grad_hm_mixed", kind="grad", prec="mixed", dets="LISA", T=2.0 ** 22, B=500, mask=ALL, tdi=20, host=False),
        # Fisher matrices of a few points (forecasts, proposal covariances)
        dict(name="fisher", kind="fisher", prec="fp64", dets="LISA", T=2.0 ** 21, B=3, mask=ALL, tdi=20, host=False),
        # relative binning in a posterior's bulk
        dict(name="hetero", kind="hetero", prec="fp64", dets="LISA", T=2.0 ** 22, B=777, mask=ALL, tdi=20, host=False),
        dict(name="hetero_mixed", kind="hetero", prec="mixed", dets="LISA+Taiji", T=2.0 ** 22, B=4096, mask=ALL, tdi=20, host=False),
        # the learned surrogate over the prior
        dict(name="surrogate_mixed", kind="surrogate", prec="mixed", dets="LISA", T=2.0 ** 22, B=8192, mask=ALL, tdi=20, host=False),
    ]


# What a unit of batch x span costs beside a unit of the FP64 likelihood (draw keeps below batch_hm).
COST = {("loglike", "fp64"): 1.0, ("plan", "fp64"): 1.0, ("loglike", "mixed"): 0.3, ("plan", "mixed"): 0.3,
        ("grad", "fp64"): 2.6, ("grad", "mixed"): 1.2, ("fisher", "fp64"): 16.0, ("hetero", "fp64"): 0.1,
        ("hetero", "mixed"): 0.05, ("surrogate", "mixed"): 0.08}
MOST = {"loglike": 1024, "plan": 512, "grad": 500, "fisher": 16, "hetero": 4096, "surrogate": 8192}


def draw(rng):
    """A case of the listed ones' ranges: every kind, precision, detector set and mode choice; spans
    from 2^18 s to 2^22 s (powers of two, the paper's 655360 s, and odd multiples of the 10 s cadence)."""
    kind, prec = rng.choice(sorted(COST))
    dets = rng.choice(["LISA", "LISA", "Taiji", "TianQin", "LISA+Taiji", NETWORK])
    if kind in ("surrogate", "hetero"):
        dets = rng.choice(["LISA", "Taiji", "LISA+Taiji"])
    span = math.exp(rng.uniform(math.log(2.0 ** 18), math.log(2.0 ** 22)))
    T = rng.choice([2.0 ** round(math.log2(span)), 655360.0, 20.0 * round(span / 20.0)])
    total = sum(T / 2 ** i for i in range(dets.count("+") + 1)) / 2.0 ** 22
    most = max(1, min(MOST[kind], int(900 / (COST[kind, prec] * total))))
    B = int(round(math.exp(rng.uniform(0.0, math.log(most)))))
    mask = ALL if kind in ("surrogate", "hetero") else rng.choice([ALL, ALL, W.MODE_22, 0x05, 0x1B])
    return dict(kind=kind, prec=prec, dets=dets, T=T, B=B, mask=mask, tdi=rng.choice([20, 20, 15]),
                host=kind in ("loglike", "grad") and B <= 64 and rng.random() < 0.5)


# ---- inputs ------------------------------------------------------------------------------------------
CONFIG = {"LISA": W.LISA, "Taiji": W.TAIJI, "TianQin": W.TIANQIN}


def grids(case):
    """[(detector description, span, first bin, bins)]: each further detector observes half the span."""
    out = []
    for i, name in enumerate(case["dets"].split("+")):
        T = case["T"] / 2 ** i
        out.append((dict(CONFIG[name], tdi_gen=case["tdi"]),) + (T,) + W.grid(T))
    return out


def shortest(case):
    return min(T for _, T, _, _ in grids(case))


def injected(case):
    return W.theta_injection(shortest(case))


# half-widths of the posterior-bulk draws around the reference, in the order of theta
BULK = np.array([20.0, 2e-4, 2e-4, 3e-4, 0.3, 0.01, 0.02, 1e-3, 1e-3, 0.01, 0.5])


def samples(case, seed):
    """Prior draws with the merger inside every span; for the heterodyned likelihood and the Fisher
    matrix, draws around the injected source; the single (2,2) point near the injected source too."""
    B, T = case["B"], shortest(case)
    rng = np.random.Generator(np.random.PCG64([seed, 1]))
    if case["kind"] == "hetero":
        return injected(case) + BULK * rng.uniform(-1.0, 1.0, (B, 11))
    if case["kind"] == "fisher" or B == 1:
        return injected(case) * (1.0 + 0.02 * rng.uniform(-1.0, 1.0, (B, 11)))
    return W.draw_prior(B, seed, T)


def data_of(case, seed):
    """Per detector (data [3][nb] complex, psd [3][nb]) on the GPU: the injected source plus noise."""
    out = []
    th = torch.tensor(injected(case), device=DEV)[None, :]
    for i, (cfg, T, k0, nb) in enumerate(grids(case)):
        f = frequencies(T, k0, nb)
        S = noise_psd(cfg, f)
        gen = torch.Generator(device=DEV)
        gen.manual_seed(1000003 * (seed + 1) + i)
        n = torch.randn((3, nb, 2), generator=gen, dtype=torch.float64, device=DEV)
        h = channels(cfg, T, th, torch.zeros(nb, dtype=torch.long, device=DEV), f, ALL)
        out.append((h + torch.view_as_complex(n) * (S * T / 4.0).sqrt(), S))
    return out


def prepare(case, seed):
    data = data_of(case, seed)
    dets = []
    for (cfg, T, k0, nb), (d, S) in zip(grids(case), data):
        det = L.Detector(cfg, T, k0, nb)
        det.set_data(torch.view_as_real(d).contiguous(), S.contiguous())
        dets.append(det)
    th = samples(case, seed)
    mask = case["mask"] | PREC[case["prec"]]
    s = dict(case=case, dets=dets, mask=mask, theta=th if case["host"] else torch.tensor(th, device=DEV))
    if case["kind"] == "plan":
        s["plan"] = L.Plan(dets, case["B"], mask, dhhh=True, autotune=False)
    elif case["kind"] == "hetero":
        ref = injected(case)
        s["hets"] = [L.Hetero(d, ref, mask, edges=coarse_edges(case, T, k0, nb)) for d, (_, T, k0, nb) in zip(dets, grids(case))]
    elif case["kind"] == "surrogate":
        s["net"] = L.Surrogate(seed=2605)
        s["net"].train(torch.tensor(W.draw_prior(8192, 2605, case["T"]), device=DEV), epochs=8, batch=1024)
    return s


def run(s):
    kind = s["case"]["kind"]
    if kind == "loglike":
        return L.loglike(s["dets"], s["theta"], s["mask"], dhhh=True, status=True)
    if kind == "plan":
        plan = s["plan"]
        plan.theta.copy_(s["theta"])
        plan.launch()
        return {"logl": plan.logl, "dhhh": plan.dhhh, "status": plan.status}
    if kind == "grad":
        if s["case"]["host"]:
            r = L.loglike_grad(s["dets"], s["theta"], s["mask"])
            return {"logl": r["logl"], "grad": r["grad"]}
        th = s["theta"].detach().requires_grad_(True)
        ll = G.loglike(th, s["dets"], s["mask"])
        (g,) = torch.autograd.grad(ll.sum(), th)
        return {"logl": ll.detach(), "grad": g}
    if kind == "fisher":
        return {"fisher": L.fisher(s["dets"], s["theta"], s["mask"])}
    if kind == "hetero":
        return L.hetero_loglike(s["hets"], s["theta"], dhhh=True, status=True)
    ll, used = s["net"].loglike(s["dets"], s["theta"], s["mask"])
    return {"logl": ll, "used": used}


# Floating-point operations that one active (sample, mode, bin) unit of the factored response cannot
# do without, and the factor of each derivative path over the value.
UNIT_FLOPS = 386.0
FACTOR = {"loglike": 1.0, "plan": 1.0, "grad": 2.5, "fisher": 11.0}


def work(case):
    B, nd, th = case["B"], len(grids(case)), samples(case, 0)
    units, table = 0.0, 0.0
    fisco = 6.0 ** -1.5 / (2.0 * math.pi * th[:, 0] * MSUN)
    for _, T, k0, nb in grids(case):
        table += nb * 3 * (16 + 8)      # the data and the noise level of each bin and channel
        for bit, (_, m) in enumerate(W.MODES):
            if case["mask"] >> bit & 1:
                units += float(np.clip(np.ceil(m * fisco * T) - k0, 0, nb).sum())
    out = B * 8.0 * {"loglike": 1 + 6 * nd, "plan": 1 + 6 * nd, "grad": 12, "fisher": 121, "hetero": 1 + 6 * nd, "surrogate": 1.5}[case["kind"]]
    if case["kind"] == "hetero":        # five modes at every edge, and the quadratic form of each bin and channel
        edges = sum(len(coarse_edges(case, T, k0, nb)) for _, T, k0, nb in grids(case))
        return {"bytes": edges * 165 * 16 + B * 88.0 + out, "flops": B * edges * (5 * UNIT_FLOPS + 3 * 15 * 30.0)}
    if case["kind"] == "surrogate":     # spline, sine and cosine and six transfer functions per unit; the network
        return {"bytes": table + B * 88.0 + out, "flops": units * 80.0 + B * 2.0 * (64 * 256 + 2 * 256 * 256 + 256 * 2560)}
    return {"bytes": table + B * 88.0 + out, "flops": units * UNIT_FLOPS * FACTOR[case["kind"]]}


# ---- the same quantities in plain 64-bit torch ----------------------------------------------------------
# arXiv:2602.12011 Sec. 2.1-2.2: TaylorF2 3.5PN modes with leading-order amplitudes, the time-frequency
# map, single-link responses on analytic orbits, frequency-domain TDI, A/E/T and the Whittle likelihood.
AU, YEAR, C, MSUN, GPC = 499.00478383615643, 31557600.0, 299792458.0, 4.925490947641267e-6, 1.02927125054339e17
EULER = 0.57721566490153286061
NORM = (1.0 / math.sqrt(2.0), 1.0 / math.sqrt(6.0), 1.0 / math.sqrt(3.0))


def frequencies(T, k0, nb):
    return torch.arange(k0, k0 + nb, dtype=torch.float64, device=DEV) / T


def noise_psd(cfg, f):
    """Equal-arm A/E/T spectra of optical-metrology and acceleration noise: [3][nb]."""
    x = 2.0 * math.pi * f * (cfg["arm_m"] / C)
    oms = (cfg["oms_m_rtHz"] * 2.0 * math.pi * f / C) ** 2
    acc = (cfg["acc_ms2_rtHz"] / (2.0 * math.pi * f * C)) ** 2
    if cfg["psd_shaping"]:
        oms = oms * (1.0 + (2e-3 / f) ** 4)
        acc = acc * (1.0 + (0.4e-3 / f) ** 2) * (1.0 + (f / 8e-3) ** 4)
    A = 8.0 * x.sin() ** 2 * ((2.0 + x.cos()) * oms + (6.0 + 4.0 * x.cos() + 2.0 * (2.0 * x).cos()) * acc)
    T = 32.0 * x.sin() ** 2 * (0.5 * x).sin() ** 2 * (oms + 4.0 * (0.5 * x).sin() ** 2 * acc)
    g = 4.0 * (2.0 * x).sin() ** 2 if cfg["tdi_gen"] == 20 else torch.ones_like(x)
    return torch.stack((A * g, A * g, T * g))


def expi(x):
    return torch.complex(x.cos(), x.sin())


def turns(x):
    """e^{2 pi i x}."""
    x = x - x.detach().round()
    return expi(2.0 * math.pi * x)


def cycles(f, tc):
    """f t_c less its nearest whole number, the product taken without rounding (Dekker's splitting)."""
    a, b = f, tc.detach()
    p = a * b
    ah, bh = a * 134217729.0, b * 134217729.0
    ah, bh = ah - (ah - a), bh - (bh - b)
    e = ((ah * bh - p) + ah * (b - bh) + (a - ah) * bh) + (a - ah) * (b - bh)
    return (p - p.round()) + e + f * (tc - tc.detach())


def per_sample(th):
    """Coefficients of the waveform and the sky frame of each sample, all [n]."""
    Mt, q, c1, c2, dL, io, ph, lam, bet, psi, tc = th.unbind(1)
    M, D = Mt * MSUN, dL * GPC
    eta, dlt, m1, m2 = q / (1.0 + q) ** 2, (q - 1.0) / (q + 1.0), q / (1.0 + q), 1.0 / (1.0 + q)
    pi = math.pi
    beta = c1 * (113.0 / 12.0 * m1 ** 2 + 25.0 / 4.0 * eta) + c2 * (113.0 / 12.0 * m2 ** 2 + 25.0 / 4.0 * eta)
    a5 = pi * (38645.0 / 756.0 - 65.0 / 9.0 * eta)
    a6 = (11583231236531.0 / 4694215680.0 - 640.0 / 3.0 * pi ** 2 - 6848.0 / 21.0 * EULER
          + (-15737765635.0 / 3048192.0 + 2255.0 / 12.0 * pi ** 2) * eta + 76055.0 / 1728.0 * eta ** 2 - 127825.0 / 1296.0 * eta ** 3)
    n = 3.0 / (128.0 * eta)
    P = [n, 0.0 * n, n * (3715.0 / 756.0 + 55.0 / 9.0 * eta), n * (-16.0 * pi + 4.0 * beta),
         n * (15293365.0 / 508032.0 + 27145.0 / 504.0 * eta + 3085.0 / 72.0 * eta ** 2 - 790.0 / 8.0 * eta * c1 * c2),
         n * a5 * (1.0 + 1.5 * math.log(6.0)), n * (a6 - 6848.0 / 21.0 * math.log(4.0)),
         n * pi * (77096675.0 / 254016.0 + 378515.0 / 1512.0 * eta - 74045.0 / 756.0 * eta ** 2)]
    sl, cl, sb, cb, sp, cp = lam.sin(), lam.cos(), bet.sin(), bet.cos(), psi.sin(), psi.cos()
    u, v = (sl, -cl, 0.0 * sl), (-sb * cl, -sb * sl, cb)
    out = dict(M=M, tc=tc, Q5=n * 3.0 * a5, Q6=n * (-6848.0 / 21.0), fisco=6.0 ** -1.5 / (2.0 * pi * M))
    out |= {"P%d" % k: P[k] for k in range(8)}
    for i in range(3):
        out["k%d" % i] = (-cb * cl, -cb * sl, -sb)[i]
        out["p%d" % i] = cp * u[i] + sp * v[i]
        out["q%d" % i] = cp * v[i] - sp * u[i]
    ci, si, c, s = io.cos(), io.sin(), (0.5 * io).cos(), (0.5 * io).sin()
    Y = {(2, 2): (math.sqrt(5 / (64 * pi)) * (1 + ci) ** 2, math.sqrt(5 / (64 * pi)) * (1 - ci) ** 2),
         (2, 1): (math.sqrt(5 / (16 * pi)) * si * (1 + ci), math.sqrt(5 / (16 * pi)) * si * (1 - ci)),
         (3, 3): (-math.sqrt(21 / (2 * pi)) * c ** 5 * s, math.sqrt(21 / (2 * pi)) * c * s ** 5),
         (3, 2): (0.5 * math.sqrt(7 / pi) * c ** 4 * (3 * ci - 2), math.sqrt(7 / (4 * pi)) * s ** 4 * (3 * ci + 2)),
         (4, 4): (3 * math.sqrt(7 / pi) * c ** 6 * s ** 2, 3 * math.sqrt(7 / pi) * c ** 2 * s ** 6)}
    mag = {(2, 2): (1.0 + 0.0 * q, 0.0, 0), (2, 1): (dlt / 3.0, -0.25, 1), (3, 3): (0.75 * math.sqrt(15 / 14) * dlt, 0.25, 1),
           (3, 2): (math.sqrt(5 / 7) / 3.0 * (1 - 3 * eta), 0.0, 2), (4, 4): (8 / 9 * math.sqrt(5 / 7) * (1 - 3 * eta), 0.5, 2)}
    for lm, (yp, yn) in Y.items():
        sg, (hm, arg, _) = (-1.0) ** lm[0], mag[lm]
        out["a%d%d" % lm] = 2.0 * pi * M ** 2 / D * (eta / (3.0 * lm[1])).sqrt() * hm
        out["h%d%d" % lm] = lm[1] * ph / (2.0 * pi) + (0.125 + arg)
        out["+%d%d" % lm] = 0.5 * (yp + sg * yn)
        out["x%d%d" % lm] = 0.5 * (sg * yn - yp)
    return out


def offsets(cfg, t):
    """Centre angle's (cos, sin) and the spacecraft offsets [3][3] (light-seconds) at t."""
    a = 2.0 * math.pi * (t / YEAR) + cfg["alpha0"]
    c, s = a.cos(), a.sin()
    arm = cfg["arm_m"] / C
    if cfg["orbit"] == 0:
        eR = arm / (2.0 * math.sqrt(3.0))
        c2, s2, out = (2 * a).cos(), (2 * a).sin(), []
        for i in range(3):
            b = 2.0 * math.pi * i / 3.0 + cfg["cartwheel0"]
            cb, sb = math.cos(b), math.sin(b)
            out.append((0.5 * eR * (c2 * cb + s2 * sb) - 1.5 * eR * cb, 0.5 * eR * (s2 * cb - c2 * sb) - 1.5 * eR * sb,
                        -math.sqrt(3.0) * eR * (c * cb + s * sb)))
        return c, s, out
    lon, lat, r = cfg["geo_lon"], cfg["geo_lat"], arm / math.sqrt(3.0)
    n = (math.cos(lat) * math.cos(lon), math.cos(lat) * math.sin(lon), math.sin(lat))
    e1 = (-math.sin(lon), math.cos(lon), 0.0)
    e2 = (n[1] * e1[2] - n[2] * e1[1], n[2] * e1[0] - n[0] * e1[2], n[0] * e1[1] - n[1] * e1[0])
    w = t / cfg["geo_period_s"]
    w = 2.0 * math.pi * (w - w.detach().round())
    out = []
    for i in range(3):
        cw, sw = (w + 2.0 * math.pi * i / 3.0).cos(), (w + 2.0 * math.pi * i / 3.0).sin()
        out.append(tuple(r * (cw * e1[j] + sw * e2[j]) for j in range(3)))
    return c, s, out


def sinc(u):
    """sin u / u, by its series where u is small (the series' last term is below 1e-19 there)."""
    small = u.abs() < 0.05
    x = torch.where(small, u, torch.zeros_like(u)) ** 2
    ser = 1 - x / 6 * (1 - x / 20 * (1 - x / 42 * (1 - x / 72 * (1 - x / 110 * (1 - x / 156)))))
    v = torch.where(small, torch.ones_like(u), u)
    return torch.where(small, ser, v.sin() / v)


def mode_channels(cfg, T, S, f, lm):
    """One mode's A/E/T signals [3][n] for the per-bin coefficients S at f."""
    pi, (l, m) = math.pi, lm
    p = {(2, 2): 0, (2, 1): 1, (3, 3): 1, (3, 2): 2, (4, 4): 2}[lm]
    key = "%d%d" % lm
    fend = m * S["fisco"]
    on = f < fend
    fs = torch.where(on, f, 0.5 * fend.detach())          # past the mode's end: any value inside, weight 0 below
    v = (2.0 * pi * S["M"] * fs / m) ** (1.0 / 3.0)
    lv = v.log()
    poly, dpoly = S["P7"], 2.0 * S["P7"]
    for k in range(6, -1, -1):
        poly, dpoly = poly * v + S["P%d" % k], dpoly * v + (k - 5.0) * S["P%d" % k]
    psi = poly / v ** 5 + lv * (S["Q5"] + S["Q6"] * v)
    dv = dpoly / v ** 5 + S["Q6"] * v * lv + S["Q5"] + S["Q6"] * v
    t = S["tc"] + m / (12.0 * pi) * dv / fs
    amp = S["a" + key] * v ** (p - 3.5)
    edge = fs > 0.9 * fend
    fe = torch.where(edge, fs, 0.95 * fend)
    z = 0.1 * fend / (fend - fe) - 0.1 * fend / (fe - 0.9 * fend)
    amp = amp * torch.where(edge, 1.0 / (1.0 + z.clamp(max=700.0).exp()), torch.ones_like(z)) * on
    c, s, dl = offsets(cfg, t)
    k, ep, eq = ([S["%s%d" % (w, i)] for i in range(3)] for w in "kpq")
    ph = S["h" + key] - cycles(fs, S["tc"]) - m / (4.0 * pi) * psi - fs * AU * (k[0] * c + k[1] * s)
    h = amp * turns(ph)
    a = pi * fs * (cfg["arm_m"] / C)
    zz = expi(-2.0 * a)
    G, sm, sp = [], [], []
    for i in range(3):                                    # links (1,2), (2,3), (3,1); third spacecraft 3, 1, 2
        r, e, o = i, (i + 1) % 3, (i + 2) % 3
        n = [dl[r][j] - dl[e][j] for j in range(3)]
        d = (n[0] ** 2 + n[1] ** 2 + n[2] ** 2).sqrt()
        kn, pn, qn = (sum(w[j] * n[j] for j in range(3)) / d for w in (k, ep, eq))
        ang = pi * fs * sum(k[j] * dl[o][j] for j in range(3))
        G.append(torch.complex(S["+" + key] * (pn ** 2 - qn ** 2), S["x" + key] * 2.0 * pn * qn) * expi(ang) * h)
        sm.append(sinc(a * (1.0 - kn)))
        sp.append(sinc(a * (1.0 + kn)))
    xyz = [G[(i + 2) % 3] * (sp[(i + 2) % 3] + zz * sm[(i + 2) % 3]) - G[i] * (sm[i] + zz * sp[i]) for i in range(3)]
    tdi = 1.0 - zz ** 2
    if cfg["tdi_gen"] == 20:
        tdi = tdi * (1.0 - zz ** 4)
    Q = tdi * torch.complex(torch.zeros_like(a), -a) * expi(-a)
    X, Y, Z = xyz
    return torch.stack((NORM[0] * Q * (Z - X), NORM[1] * Q * (X - 2.0 * Y + Z), NORM[2] * Q * (X + Y + Z)))


def channels(cfg, T, th, si, f, mask):
    """The signal's A/E/T channels [3][n] at frequencies f of the samples th[si]."""
    S = {k: v[si] for k, v in per_sample(th).items()}
    return sum(mode_channels(cfg, T, S, f, lm) for bit, lm in enumerate(W.MODES) if mask >> bit & 1)


def active(case, th, T, k0, nb, most):
    """Chunks (sample index, bin index) of every sample's bins below its last mode's end."""
    top = max(m for bit, (_, m) in enumerate(W.MODES) if case["mask"] >> bit & 1)
    end = np.clip(np.ceil(top * 6.0 ** -1.5 / (2.0 * math.pi * th[:, 0] * MSUN) * T) - k0 + 1, 1, nb).astype(np.int64)
    lo = 0
    while lo < len(end):
        hi = lo + max(1, int(np.searchsorted(np.cumsum(end[lo:]), most)))
        n = torch.tensor(end[lo:hi], device=DEV)
        si = torch.repeat_interleave(torch.arange(lo, min(hi, len(end)), device=DEV), n)
        bi = torch.arange(len(si), device=DEV) - torch.repeat_interleave(n.cumsum(0) - n, n)
        yield si, bi
        lo = hi


def exact(case, seed):
    if case["kind"] == "surrogate":
        return None      # the network and its splines stand for the likelihood, to about 1e-3 of the signal
    if case["kind"] == "hetero":
        return exact_hetero(case, seed)
    x, data = samples(case, seed), data_of(case, seed)
    B, nd = case["B"], len(data)
    th = torch.tensor(x, device=DEV)
    ll = torch.zeros(B, dtype=torch.float64, device=DEV)
    dhhh = torch.zeros((B, nd, 3, 2), dtype=torch.float64, device=DEV)
    grad = torch.zeros((B, 11), dtype=torch.float64, device=DEV)
    F = torch.zeros((B, 11, 11), dtype=torch.float64, device=DEV)
    for I, ((cfg, T, k0, nb), (d, S)) in enumerate(zip(grids(case), data)):
        f, w = frequencies(T, k0, nb), 4.0 / (S * T)
        ll -= 0.5 * (w * (d.real ** 2 + d.imag ** 2)).sum()
        for si, bi in active(case, x, T, k0, nb, 1 << (19 if case["kind"] == "grad" else 21)):
            fb, wb, db = f[bi], w[:, bi], d[:, bi]
            if case["kind"] == "fisher":
                J = []
                for i in range(11):
                    with torch.autograd.forward_ad.dual_level():
                        e = torch.zeros_like(th)
                        e[:, i] = 1.0
                        h = channels(cfg, T, torch.autograd.forward_ad.make_dual(th, e), si, fb, case["mask"])
                        J.append(torch.autograd.forward_ad.unpack_dual(h).tangent)
                for i in range(11):
                    for j in range(i, 11):
                        F[:, i, j].index_add_(0, si, (wb * (J[i].real * J[j].real + J[i].imag * J[j].imag)).sum(0))
                continue
            v = th.clone().requires_grad_(case["kind"] == "grad")
            h = channels(cfg, T, v, si, fb, case["mask"])
            dh, hh = wb * (db.real * h.real + db.imag * h.imag), wb * (h.real ** 2 + h.imag ** 2)
            if case["kind"] == "grad":
                grad += torch.autograd.grad((dh - 0.5 * hh).sum(), v)[0]
            for c in range(3):
                dhhh[:, I, c, 0].index_add_(0, si, dh[c].detach())
                dhhh[:, I, c, 1].index_add_(0, si, hh[c].detach())
    ll += (dhhh[..., 0] - 0.5 * dhhh[..., 1]).sum((1, 2))
    if case["kind"] == "fisher":
        return {"fisher": F.triu() + F.triu(1).transpose(1, 2)}
    if case["kind"] == "grad":
        return {"logl": ll, "grad": grad}
    return {"logl": ll, "dhhh": dhhh, "status": None}


# ---- relative binning -----------------------------------------------------------------------------------
def taper_marks(case, T, k0, m):
    """Bins of the fractions 1 - 0.1 * 0.7^j (j = 0..10) of the reference's m F_isco, and the last bin below it."""
    fe = m * 6.0 ** -1.5 / (2.0 * math.pi * injected(case)[0] * MSUN)
    return [math.ceil((1.0 - 0.1 * 0.7 ** j) * fe * T) - k0 for j in range(11)], math.ceil(fe * T) - k0 - 1


def coarse_edges(case, T, k0, nb):
    """Coarse-bin edges: uniform in the relative-binning phase metric up to the band end, plus the marks
    of each mode's taper (none between a mode's last mark and its end)."""
    ms = [m for bit, (_, m) in enumerate(W.MODES) if case["mask"] >> bit & 1]
    kmax = min(nb - 1, max(taper_marks(case, T, k0, m)[1] for m in ms))
    f = np.arange(k0, k0 + kmax + 1) / T
    metric = sum(np.sign(g) * (f / (f[0] if g < 0 else f[-1])) ** g for g in (-5 / 3, -2 / 3, 1.0, 5 / 3, 7 / 3))
    cand = set(np.searchsorted(metric, np.linspace(metric[0], metric[-1], HET_BINS + 1)[1:-1]).tolist()) | {0, kmax}
    for m in ms:
        cand |= set(taper_marks(case, T, k0, m)[0])
    ends = [(taper_marks(case, T, k0, m)[0][-1], taper_marks(case, T, k0, m)[1]) for m in ms]
    return np.array(sorted(k for k in cand if 0 <= k <= kmax and (k == kmax or not any(a < k <= b for a, b in ends))), dtype=np.int64)


def exact_hetero(case, seed):
    x, B, grid = samples(case, seed), case["B"], grids(case)
    ll = torch.zeros(B, dtype=torch.float64, device=DEV)
    dhhh = torch.zeros((B, len(grid), 3, 2), dtype=torch.float64, device=DEV)
    th, ref = torch.tensor(x, device=DEV), torch.tensor(injected(case), device=DEV)[None, :]
    for I, ((cfg, T, k0, nb), (d, S)) in enumerate(zip(grid, data_of(case, seed))):
        e = torch.tensor(coarse_edges(case, T, k0, nb), device=DEV)
        ne, K = len(e), int(e[-1]) + 1
        f, w = frequencies(T, k0, nb), 4.0 / (S * T)
        ll -= 0.5 * (w * (d.real ** 2 + d.imag ** 2)).sum()
        S0 = {k: v.expand(K) for k, v in per_sample(ref).items()}
        h0 = torch.stack([mode_channels(cfg, T, S0, f[:K], lm) for lm in W.MODES])     # [mode][channel][bin]
        b = (torch.searchsorted(e, torch.arange(K, device=DEV), right=True) - 1).clamp(max=ne - 2)
        df = f[:K] - f[e][b]

        def sums(y):
            out = torch.zeros(y.shape[:-1] + (ne - 1,), dtype=torch.complex128, device=DEV)
            return out.index_add_(y.dim() - 1, b, y)
        A = [sums(w[:, :K] * d[:, :K].conj() * h0 * df ** o) for o in range(2)]
        Bs = [sums(w[:, :K] * h0[:, None] * h0[None].conj() * df ** o) for o in range(3)]
        last = torch.tensor([taper_marks(case, T, k0, m)[0][-1] for _, m in W.MODES], device=DEV)
        use = (e[None, None, :] <= last[:, None, None]) & (h0[:, :, e] != 0)
        src = torch.where(use, torch.arange(ne, device=DEV), -1).cummax(2).values
        step = 256
        for lo in range(0, B, step):
            n = min(step, B - lo)
            Ss = {k: v.repeat_interleave(ne) for k, v in per_sample(th[lo:lo + n]).items()}
            h = torch.stack([mode_channels(cfg, T, Ss, f[e].repeat(n), lm).reshape(3, n, ne) for lm in W.MODES])
            r = h / torch.where(use, h0[:, :, e], torch.ones_like(h0[:, :, e]))[:, :, None, :]
            r = r.gather(3, src.clamp(min=0)[:, :, None, :].expand(-1, -1, n, -1)) * (src >= 0)[:, :, None, :]
            r0 = r[..., :-1]
            r1 = (r[..., 1:] - r0) / (f[e[1:]] - f[e[:-1]])
            dh = (A[0][:, :, None] * r0 + A[1][:, :, None] * r1).real.sum((0, 3))
            hh = torch.zeros_like(dh)
            for i in range(5):
                for j in range(5):
                    hh += (Bs[0][i, j][:, None] * r0[i] * r0[j].conj() + Bs[2][i, j][:, None] * r1[i] * r1[j].conj()
                           + Bs[1][i, j][:, None] * (r1[i] * r0[j].conj() + r0[i] * r1[j].conj())).real.sum(2)
            dhhh[lo:lo + n, I, :, 0], dhhh[lo:lo + n, I, :, 1] = dh.T, hh.T
    ll += (dhhh[..., 0] - 0.5 * dhhh[..., 1]).sum((1, 2))
    return {"logl": ll, "dhhh": dhhh, "status": None}
