"""GPU tests of the FP64 path's fixed-point unit (pe_device_fx.cuh) where it can go wrong: both sides of the
rule that picks it (a = pi f L against 4, the arm's eccentricity), both orbits, merger times on either side
of zero, samples whose lowest mode is alone or vanishes inside a tile, and edges of 128-bin tiles.

Tolerances: the FP64 parity bars of tests/_helpers.py (1e-10 of each quantity's scale plus the rounding
floor both sides compute in); the unit's own errors are a few 2^-56 of unit-sized quantities, far below.
"""
import numpy as np
import pytest

import tests._helpers as H
from paper_2602_12011_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def Lb():
    from paper_2602_12011_gb300 import _lib
    _lib.lib()
    return _lib


@pytest.fixture(scope="module")
def oracle_mod():
    from oracle import oracle as O
    O.build()
    return O


# (detector, span, first bin, bins): a = pi f L at the last bin just below and above 4 for the LISA and
# TianQin arms (the general unit takes over), an arm whose eccentricity is above the unit's bound, one-bin
# and tile-edge grids
GRIDS = {
    "lisa_a_below_4": (W.LISA, 2.0 ** 14, 2300, 190),
    "lisa_a_above_4": (W.LISA, 2.0 ** 14, 2300, 300),
    "tianqin_a_below_4": (W.TIANQIN, 2.0 ** 11, 4450, 140),
    "tianqin_a_above_4": (W.TIANQIN, 2.0 ** 11, 4450, 250),
    "long_arm": (dict(W.LISA, arm_m=3.0e10), 2.0 ** 16, 7, 400),
    "tdi15_odd_span": (dict(W.TAIJI, tdi_gen=15), 65536.0 - 321.7, 7, 129),
    "one_bin": (W.LISA, 2.0 ** 16, 200, 1),
    "tile_edge": (W.TAIJI, 2.0 ** 16, 7, 128),
}


def _samples(T, fmax):
    """Masses whose modes end inside and beyond the grid, the single odd and even modes' corners (q = 1
    drops the odd modes), merger times before, inside and after the span."""
    fisco1 = 6.0 ** -1.5 / (2.0 * np.pi * 4.925490947641267e-6)     # of one solar mass
    th = W.draw_prior(8, 17, T)
    th[:, 0] = np.clip(fisco1 * np.array([0.6, 1.3, 1.9, 2.2, 3.1, 3.9, 4.2, 9.0]) / fmax, 1e3, 1e9)
    th[2, 1] = 1.0
    th[3, 10] = -0.3 * T
    th[4, 10] = 0.0
    th[5, 10] = 1.7 * T
    return th


@pytest.mark.parametrize("mask", [W.MODE_ALL, 0x10, 0x09])
@pytest.mark.parametrize("name", sorted(GRIDS))
def test_fixed_point_unit_parity(oracle_mod, Lb, name, mask):
    det, T, k0, nb = GRIDS[name]
    fmax = (k0 + nb - 1) / T
    th = _samples(T, fmax)
    od = H.oracle_detector(oracle_mod, det, T, k0, nb, th[0], mask, 23)
    gd = H.library_detector(Lb, od)
    g = Lb.loglike([gd], th, mask, dhhh=True)
    ll, dhhh = oracle_mod.loglike_batch([od], th, mask)
    dd = np.array([oracle_mod.loglike([od], th[0], 0)["dd"][0]])
    H.assert_loglike_parity(g, ll, dhhh, dd, H.floor_terms(oracle_mod, [od], th, mask))


@pytest.mark.parametrize("mask", [W.MODE_ALL, 0x12, 0x08])
@pytest.mark.parametrize("det,T", [(W.LISA, 2.0 ** 16), (W.TIANQIN, 2.0 ** 15), (dict(W.LISA, arm_m=3.0e10), 2.0 ** 14)])
def test_gradient_where_weights_and_modes_vanish(oracle_mod, Lb, det, T, mask):
    """The gradient's fixed-point sweep (and the general one, for the long arm) on the bars of the gradient parity
    tests, where polarisation weights vanish but their derivatives do not (face-on, face-off), at the
    poles, at edge-on, with equal masses, and with the merger before the data; both precisions."""
    k0, nb = W.grid(T)
    inj = W.theta_injection(T)
    od = H.oracle_detector(oracle_mod, det, T, k0, nb, inj, W.MODE_ALL, 29)
    gd = H.library_detector(Lb, od)
    th = W.draw_prior(6, 19, T)
    th[0, 5], th[1, 5], th[2, 5] = 0.0, np.pi, 0.5 * np.pi
    th[0, 8], th[3, 8] = 0.5 * np.pi, -0.5 * np.pi
    th[4, 1] = 1.0 + 1e-9
    th[5, 10] = -0.2 * T
    for flag in (0, Lb.PE_PREC_MIXED):
        g = Lb.loglike_grad([gd], th, mask | flag)
        for s in range(th.shape[0]):
            r = oracle_mod.loglike([od], th[s], mask)
            ll, ref = oracle_mod.grad([od], th[s], mask)
            F = oracle_mod.fisher([od], th[s], mask)
            assert abs(g["logl"][s] - ll) <= 1e-10 * H.scale_of(r["dh"], r["hh"], r["dd"])
            for i in range(11):
                tol = H.grad_tolerance(ref[i], float(np.sum(r["hh"])), F[i, i])
                assert abs(g["grad"][s, i] - ref[i]) <= tol, (flag, s, W.PARAM_NAMES[i], g["grad"][s, i], ref[i], tol)


# High masses, unequal and spinning: t_f's series terms are hundreds of times their sum, whose double word is far from normalised.
CANCELLING = np.array([
    [9.44096895e+06, 9.11190755, -0.836978605, -0.425334183, 27.3127246, 2.56475767, 4.65730762, 2.08844287, -0.279393, 2.21142, 505558.0],
    [9.99833e+06, 7.88270, -0.624269, -0.926790, 35.2661, 1.04696, 2.18150, 1.61548, -0.313205, 2.70229, 353475.0],
    [9.75437e+06, 9.77584, -0.834856, -0.392306, 7.79320, 1.67881, 1.96344, 4.23071, -0.428794, 1.96235, 356152.0],
    [9.78440e+06, 9.64430, -0.920518, 0.585617, 31.5393, 0.821924, 0.508002, 0.761395, -0.0310906, 2.33068, 317660.0]])


@pytest.mark.parametrize("first", range(66, 600, 89))
def test_time_far_below_its_terms(oracle_mod, Lb, first):
    T, nb = 655360.0, 89
    od = H.oracle_detector(oracle_mod, W.LISA, T, first, nb, CANCELLING[0], 0x10, 37)
    gd = H.library_detector(Lb, od)
    th = np.repeat(CANCELLING, 64, axis=0)
    th[:, 0] *= 1.0 + 1e-4 * np.tile(np.arange(64), len(CANCELLING))
    g = Lb.loglike([gd], th, 0x10, dhhh=True)
    ll, dhhh = oracle_mod.loglike_batch([od], th, 0x10)
    dd = np.array([oracle_mod.loglike([od], th[0], 0)["dd"][0]])
    H.assert_loglike_parity(g, ll, dhhh, dd, H.floor_terms(oracle_mod, [od], th, 0x10))


@pytest.mark.parametrize("nb,copies", [(1, 1), (32, 1), (33, 1), (129, 1), (160, 2000)])
@pytest.mark.parametrize("det,mask", [(W.LISA, W.MODE_ALL), (W.TIANQIN, 0x19), (dict(W.TAIJI, tdi_gen=15), 0x08)])
def test_fisher_at_pass_and_tile_edges(oracle_mod, Lb, det, mask, nb, copies):
    """Grids around the 32-bin pass and the 128-bin tile, masses whose modes end inside them, whole tiles per item
    (copies: many points) as well as quarters; on the bar of the Fisher parity test, 1e-10 of sqrt(F_ii F_kk)."""
    T, k0 = 2.0 ** 16, 30
    th = _samples(T, (k0 + nb - 1) / T)
    od = H.oracle_detector(oracle_mod, det, T, k0, nb, th[0], W.MODE_ALL, 41)
    F = Lb.fisher([H.library_detector(Lb, od)], np.tile(th, (copies, 1)), mask)
    for s in range(len(th)):
        Fr = oracle_mod.fisher([od], th[s], mask)
        d = np.sqrt(np.abs(np.outer(np.diag(Fr), np.diag(Fr))))
        assert np.all(np.abs(F[s] - Fr) <= 1e-10 * d + 1e-300), (s, np.max(np.abs(F[s] - Fr) / (d + 1e-300)))
    np.testing.assert_array_equal(F, np.tile(F[:len(th)], (copies, 1, 1)))


def test_surrogate_bins_below_the_first_node(Lb):
    """The FP64 surrogate's fixed-point phase spline where the grid begins on the first node (1e-4 Hz), a fraction of an interval
    below it and far below it (extrapolated in FP64), against the mixed unit's double-word spline on the same nodes;
    bar: that pair's own, 1e-6 of the log-likelihood's terms."""
    import torch
    T = 2.0 ** 18
    net = Lb.Surrogate(seed=5)
    net.train(torch.tensor(W.draw_prior(1024, 5, T), device="cuda"), epochs=1, batch=1024)
    net.set_node_source(1)
    th = W.draw_prior(512, 6, T)
    th = torch.tensor(th[(th[:, 1] <= 8.0) & (th[:, 0] >= 3e5)][:64], device="cuda")
    rng = np.random.default_rng(7)
    for f0 in (1e-4, 0.997e-4, 0.9e-4):
        k0, nb = int(np.ceil(f0 * T)), 300
        det = Lb.Detector(W.LISA, T, k0, nb)
        det.set_data(torch.tensor(1e-21 * rng.standard_normal((3, nb, 2)), device="cuda"),
                     torch.full((3, nb), 1e-38, dtype=torch.float64, device="cuda"))
        a = net.loglike([det], th, W.MODE_ALL)[0].cpu().numpy()
        b = net.loglike([det], th, W.MODE_ALL | Lb.PE_PREC_MIXED)[0].cpu().numpy()
        r = Lb.loglike([det], th, W.MODE_ALL, dhhh=True)["dhhh"].cpu().numpy()
        scale = 0.5 * det.data_norm().sum() + np.abs(r[..., 0].sum(axis=(1, 2))) + 0.5 * r[..., 1].sum(axis=(1, 2))
        assert np.all(np.isfinite(a)) and np.all(np.abs(a - b) <= 1e-6 * scale), (f0, np.max(np.abs(a - b) / scale))


@pytest.mark.parametrize("nbins,mask", [(1, 0x04), (2, W.MODE_ALL), (64, W.MODE_ALL), (300, 0x19)])
def test_heterodyned_ratios_on_either_side_of_the_bound(oracle_mod, Lb, nbins, mask):
    """The fixed-point contraction and its FP64 fallback: distances that put every ratio far below, just below, just above and far
    above 2, with and without shifts in the other parameters, one to 300 coarse bins; on the bar of the
    heterodyned parity tests, against the oracle on the same edges."""
    from oracle import hetero as HT
    T = 2.0 ** 19
    k0, nb = W.grid(T)
    th0 = W.theta_injection(T)
    od = H.oracle_detector(oracle_mod, W.LISA, T, k0, nb, th0, mask, 47)
    gd = H.library_detector(Lb, od)
    edges = HT.default_edges(T, k0, nb, th0, mask, nbins)
    oh = HT.Hetero(od, th0, mask, edges)
    gh = Lb.Hetero(gd, th0, mask, edges=edges)
    th = np.tile(th0, (14, 1))
    th[:, 4] /= np.tile([0.02, 0.9, 1.9, 1.999999, 2.000001, 2.1, 40.0], 2)
    th[7:, 0] *= 1.00003
    th[7:, 7] += 0.004
    th[7:, 10] += 0.7
    g = Lb.hetero_loglike([gh], th, dhhh=True)
    for s in range(len(th)):
        r = oh.loglike(th[s])
        scale = H.scale_of(r["dh"], r["hh"], r["dd"])
        assert abs(g["logl"][s] - r["logl"]) <= 1e-10 * scale, (s, abs(g["logl"][s] - r["logl"]) / scale)
        assert np.all(np.abs(g["dhhh"][s, 0] - np.stack([r["dh"], r["hh"]], -1)) <= 1e-10 * scale)


def test_a_bin_without_a_finite_datum(Lb):
    """One NaN among the data: the likelihood, every gradient component and the heterodyned sums of its channel are NaN for the
    samples that reach the bin, as in floating point, and the others' values do not change."""
    T = 2.0 ** 17
    k0, nb = W.grid(T)
    th = W.draw_prior(2, 3, T)
    th[:, 0] = [3e6, 3e5]      # the first ends below 1.5e-3 Hz * 4/2, the second well above
    rng = np.random.default_rng(5)
    d = 1e-21 * (rng.standard_normal((3, nb)) + 1j * rng.standard_normal((3, nb)))
    psd = np.full((3, nb), 1e-38)
    bad = int(0.01 * T) - k0
    out = []
    for value in (d[1, bad], np.nan):
        d[1, bad] = value
        det = Lb.Detector(W.LISA, T, k0, nb)
        det.set_data(d, psd)
        het = Lb.Hetero(det, th[1], W.MODE_ALL, nbins_coarse=32)
        out.append((Lb.loglike([det], th, W.MODE_ALL, dhhh=True)["dhhh"], Lb.loglike_grad([det], th, W.MODE_ALL)["grad"],
                    Lb.hetero_loglike([het], th[1:], dhhh=True)["dhhh"]))
    (l0, g0, h0), (l1, g1, h1) = out
    np.testing.assert_array_equal(l1[0], l0[0])
    np.testing.assert_array_equal(g1[0], g0[0])
    assert np.isnan(l1[1, 0, 1, 0]) and np.all(np.isnan(g1[1])) and np.isnan(h1[0, 0, 1, 0])
    np.testing.assert_array_equal(l1[1, 0, [0, 2]], l0[1, 0, [0, 2]])
    np.testing.assert_array_equal(h1[0, 0, [0, 2]], h0[0, 0, [0, 2]])


@pytest.mark.parametrize("det", [W.LISA, dict(W.LISA, arm_m=3.0e10)], ids=["fixed_point", "general"])
def test_fisher_of_a_point_does_not_depend_on_the_batch(Lb, det):
    """A point's Fisher matrix is the same bits alone and inside batches from one tile per SM to more than a thousand tiles
    per SM, on both sides of the rule that picks the kernel's work items."""
    T = 2.0 ** 16
    k0, nb = W.grid(T)
    d = Lb.Detector(det, T, k0, nb)
    d.inject(W.theta_injection(T), W.MODE_ALL, W.normals(nb, 2))
    th = _samples(T, 0.02)
    alone = np.concatenate([Lb.fisher([d], t[None, :], W.MODE_ALL) for t in th])
    for B in (8, 72, 1200, 8000):
        np.testing.assert_array_equal(Lb.fisher([d], np.tile(th, (B // 8, 1)), W.MODE_ALL), np.tile(alone, (B // 8, 1, 1)))


@pytest.mark.parametrize("arm_m", [2.5e9, 3.0e10], ids=["fixed_point", "general"])
def test_amplitudes_at_the_limits_of_a_double(Lb, arm_m):
    """A distance so small that the amplitude or <h|h> overflows gives no finite log L or derivative in the distance, in every
    unit and on the surrogate's spline path; one so large that the signal underflows gives the log L of no signal."""
    import torch
    T = 2.0 ** 16
    d = Lb.Detector(dict(W.LISA, arm_m=arm_m), T, 200, 300)
    rng = np.random.default_rng(3)
    d.set_data(1e-21 * (rng.standard_normal((3, 300)) + 1j * rng.standard_normal((3, 300))), np.full((3, 300), 1e-38))
    none = -0.5 * d.data_norm().sum()
    th0 = np.array([1e6, 2.0, 0.1, -0.2, 1.0, 0.6, 0.9, 2.0, 0.4, 1.1, 100.0])
    th = np.tile(th0, (8, 1))
    th[:, 4] = [5e-324, 1e-312, 1e-306, 1e-290, 1e-200, 1e-160, 1e280, 1e290]
    net = Lb.Surrogate(seed=1)
    net.set_node_source(1)
    for flag in (0, Lb.PE_PREC_MIXED):
        for mask in (W.MODE_22, W.MODE_ALL):
            ll = Lb.loglike([d], th, mask | flag)["logl"]
            g = Lb.loglike_grad([d], th, mask | flag)
            sur = net.loglike([d], torch.tensor(th, device="cuda"), mask | flag)[0].cpu().numpy()
            for x in (ll, g["logl"], g["grad"][:, 4], sur):
                assert not np.any(np.isfinite(x[:6])), (flag, mask, x)
            assert not np.any(np.isfinite(d.signal(th[0], mask | flag)[:, :60]))    # below the (2,2) mode's end
            for x in (ll, g["logl"], sur):
                assert np.all(np.abs(x[6:] - none) <= 1e-12 * abs(none)), (flag, mask, x)
            assert np.all(np.isfinite(g["grad"][6:]))
    het = Lb.Hetero(d, th0, W.MODE_ALL, nbins_coarse=20)
    ll = Lb.hetero_loglike([het], th)["logl"]
    assert not np.any(np.isfinite(ll[:6])) and np.all(np.abs(ll[6:] - none) <= 1e-12 * abs(none)), ll
