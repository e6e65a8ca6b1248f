"""The general kernels on detectors that do not take the fixed-point unit (an arm whose orbital eccentricity is
above the unit's bound, and a grid with pi f L above 4), alone and beside a LISA, which sends the whole
call there: the per-bin signal, the likelihood in both precisions, Fisher matrices, the heterodyned
likelihood, the surrogate's log-likelihood and mismatch, tuned launches and the checked build. The
bars are those of the same quantities' tests on the other detectors."""
import os

import numpy as np
import pytest

from paper_2602_12011_gb300 import workloads as W
from tests import _helpers as H

pytestmark = pytest.mark.gpu

LONG = dict(W.LISA, arm_m=3.0e10)


@pytest.fixture(scope="module")
def Lb(tmp_path_factory):
    import torch
    assert torch.cuda.is_available(), "GPU tests need CUDA"
    os.environ["PE_TUNE_CACHE"] = str(tmp_path_factory.mktemp("tune") / "tune.json")
    from paper_2602_12011_gb300 import build as B
    from paper_2602_12011_gb300 import _lib
    B.build()
    _lib.lib()
    return _lib


# detector, span, first bin, bins of each member
SETS = {
    "long_arm": [(LONG, 2.0 ** 15, 4, 700)],
    "a_above_4": [(W.LISA, 2.0 ** 14, 2300, 300)],
    "tianqin_a_above_4": [(W.TIANQIN, 2.0 ** 11, 4450, 250)],
    "lisa_and_long_arm": [(W.LISA, 2.0 ** 15, 4, 700), (dict(LONG, tdi_gen=15), 2.0 ** 14, 7, 389)],
}


def _members(O, Lb, name, noise=31):
    inj = np.array([1e6, 2.0, 0.5, 0.3, 25.8, 0.4, 1.3, 1.375, -1.2108, 2.659, 0.4 * 2.0 ** 14])
    ods = [H.oracle_detector(O, det, T, k0, nb, inj, W.MODE_ALL, noise + i) for i, (det, T, k0, nb) in enumerate(SETS[name])]
    dd = np.array([O.loglike([od], inj, 0)["dd"][0] for od in ods])
    return ods, [H.library_detector(Lb, od) for od in ods], dd


def _theta(name, n=7, seed=17):
    """Prior samples whose taper ends lie across the first member's grid."""
    det, T, k0, nb = SETS[name][0]
    th = W.draw_prior(n, seed, 2.0 ** 14)
    fisco1 = 6.0 ** -1.5 / (2.0 * np.pi * 4.925490947641267e-6)
    th[:, 0] = np.clip(fisco1 * np.linspace(0.6, 6.0, n) * T / (k0 + nb), 1e3, 1e9)
    th[1, 1] = 1.0
    th[2, 10] = -0.3 * T
    return th


@pytest.mark.parametrize("mix", [False, True], ids=["fp64", "mixed"])
@pytest.mark.parametrize("mask", [W.MODE_ALL, 0x12])
@pytest.mark.parametrize("name", sorted(SETS))
def test_likelihood(oracle_mod, Lb, name, mask, mix):
    ods, gds, dd = _members(oracle_mod, Lb, name)
    th = _theta(name)
    flag = Lb.PE_PREC_MIXED if mix else 0
    g = Lb.loglike(gds, th, mask | flag, dhhh=True)
    ll, dhhh = oracle_mod.loglike_batch(ods, th, mask)
    Q = H.floor_terms(oracle_mod, ods, th, mask)
    H.assert_loglike_parity(g, ll, dhhh, dd, Q, u=H.U_DW if mix else H.U64, name="general:%s:%s" % (name, mix))
    one = Lb.loglike(gds, th[3:4], mask | flag, dhhh=True)
    np.testing.assert_array_equal(one["dhhh"][0], g["dhhh"][3])
    np.testing.assert_array_equal(one["logl"], g["logl"][3:4])


@pytest.mark.parametrize("mix", [False, True], ids=["fp64", "mixed"])
@pytest.mark.parametrize("name", ["long_arm", "a_above_4", "tianqin_a_above_4"])
def test_signal(oracle_mod, Lb, name, mix):
    (det, T, k0, nb), = SETS[name]
    f = H.grid_f(T, k0, nb)
    d = Lb.Detector(det, T, k0, nb)
    for th in _theta(name, 3):
        h = d.signal(th, W.MODE_ALL | (Lb.PE_PREC_MIXED if mix else 0))
        H.assert_signal_parity(h, oracle_mod.response(det, th, W.MODE_ALL, f), "general_signal:" + name,
                               H.phase_magnitude(oracle_mod, th, W.MODE_ALL, f), u=H.U_DW if mix else H.U64)


@pytest.mark.parametrize("mask", [W.MODE_ALL, 0x19, 0x04])
@pytest.mark.parametrize("name", sorted(SETS))
def test_fisher(oracle_mod, Lb, name, mask):
    ods, gds, _ = _members(oracle_mod, Lb, name)
    th = _theta(name, 4)
    F = Lb.fisher(gds, th, mask)
    for s in range(len(th)):
        Fr = oracle_mod.fisher(ods, th[s], mask)
        d = np.sqrt(np.abs(np.outer(np.diag(Fr), np.diag(Fr))))
        assert np.all(np.abs(F[s] - Fr) <= 1e-10 * d + 1e-300), (s, np.max(np.abs(F[s] - Fr) / (d + 1e-300)))


@pytest.mark.parametrize("mix", [False, True], ids=["fp64", "mixed"])
@pytest.mark.parametrize("nbins", [48, 300])
@pytest.mark.parametrize("name", ["long_arm", "lisa_and_long_arm"])
def test_heterodyned(oracle_mod, Lb, name, nbins, mix):
    from oracle import hetero as HT
    th0 = np.array([8e5, 2.0, 0.4, -0.2, 20.0, 0.6, 0.9, 2.0, 0.4, 1.1, 0.4 * 2.0 ** 14])
    ods, gds, _ = _members(oracle_mod, Lb, name)
    edges = [HT.default_edges(od.T, od.k0, od.nb, th0, W.MODE_ALL, nbins) for od in ods]
    ohs = [HT.Hetero(od, th0, W.MODE_ALL, e) for od, e in zip(ods, edges)]
    ghs = [Lb.Hetero(gd, th0, W.MODE_ALL | (Lb.PE_PREC_MIXED if mix else 0), edges=e) for gd, e in zip(gds, edges)]
    th = np.tile(th0, (7, 1))
    th[1:, 0] *= 1.001
    th[2:, 4] /= [0.02, 1.9, 2.1, 40.0, 1.0]
    th[4:, 7] += 0.01
    th[6, 5] = 1.4
    g = Lb.hetero_loglike(ghs, th, dhhh=True)
    Q = H.floor_terms(oracle_mod, ods, th, W.MODE_ALL)
    for s in range(len(th)):
        r = HT.loglike_network(ohs, th[s])
        H.assert_loglike_parity({"logl": g["logl"][s:s + 1], "dhhh": g["dhhh"][s:s + 1]}, np.array([r["logl"]]),
                                np.stack([r["dh"], r["hh"]], -1).reshape(1, len(ods), 3, 2), r["dd"], Q[s],
                                u=H.U_DW if mix else H.U64, name="general_hetero:%s:%s" % (name, mix))


@pytest.mark.parametrize("mix", [False, True], ids=["fp64", "mixed"])
@pytest.mark.parametrize("dets", [[LONG], [W.LISA, LONG]], ids=["long_arm", "lisa_and_long_arm"])
def test_surrogate(oracle_mod, Lb, dets, mix):
    """The spline path from the plain generator's node values within 1e-6 of the likelihood's scale of the oracle, samples
    outside its box on the per-bin path bit for bit, and the mismatch of both: that of the spline alone inside the box, 0 outside."""
    import torch
    T = 2.0 ** 19
    k0, nb = W.grid(T)
    inj = np.array([2e6, 3.0, 0.5, 0.3, 25.8, 0.4, 1.3, 1.375, -1.2108, 2.659, 0.8 * T])
    ods = [H.oracle_detector(oracle_mod, det, T, k0, nb, inj, W.MODE_ALL, 5 + i) for i, det in enumerate(dets)]
    gds = [H.library_detector(Lb, od) for od in ods]
    s = Lb.Surrogate(seed=1)
    s.set_node_source(1)
    th = np.vstack([inj, W.draw_prior(7, 31, T)])
    th[1:, 0] = np.linspace(5e5, 9e6, 7)
    th[1:, 1] = np.minimum(th[1:, 1], 8.0)
    th[6:, 1] = 10.5                              # outside the box
    tt = torch.tensor(th, device="cuda")
    flag = Lb.PE_PREC_MIXED if mix else 0
    ll, used = s.loglike(gds, tt, W.MODE_ALL | flag)
    ll = ll.cpu().numpy()
    np.testing.assert_array_equal(used.cpu().numpy(), [1] * 6 + [0] * 2)
    ref, dhhh = oracle_mod.loglike_batch(ods, th, W.MODE_ALL)
    dd = sum(oracle_mod.loglike([od], inj, 0)["dd"].sum() for od in ods)
    scale = 0.5 * dd + np.abs(dhhh[..., 0].sum(axis=(1, 2))) + 0.5 * dhhh[..., 1].sum(axis=(1, 2))
    assert np.all(np.abs(ll - ref) <= 1e-6 * scale), np.abs(ll - ref) / scale
    np.testing.assert_array_equal(ll[6:], Lb.loglike(gds, th, W.MODE_ALL | flag)["logl"][6:])
    if not mix:
        mm = s.mismatch(gds[-1], tt, W.MODE_ALL).cpu().numpy()
        assert np.all(mm[:6] <= 1e-5) and np.all(mm[:6] >= 0.0) and np.all(mm[6:] == 0.0), mm
    s.close()


@pytest.mark.parametrize("mix", [False, True], ids=["fp64", "mixed"])
def test_every_tuning_choice_gives_the_same_bits(Lb, mix):
    dets = []
    for i, (det, T, k0, nb) in enumerate(SETS["lisa_and_long_arm"]):
        d = Lb.Detector(det, T, k0, nb)
        d.inject(W.theta_injection(2.0 ** 14), W.MODE_ALL, W.normals(nb, 5 + i))
        dets.append(d)
    th = W.draw_prior(37, 21, 2.0 ** 14)
    m = W.MODE_ALL | (Lb.PE_PREC_MIXED if mix else 0)
    ref = Lb.loglike(dets, th, m, dhhh=True)
    for r in (1, 2, 4, 8):
        for v, c in ((0, 16), (1, 2), (2, 8)):
            Lb.pe_tune_set([d.handle for d in dets], len(th), m, v, c, r)
            out = Lb.loglike(dets, th, m, dhhh=True)
            np.testing.assert_array_equal(out["logl"], ref["logl"])
            np.testing.assert_array_equal(out["dhhh"], ref["dhhh"])


def test_checked_build(oracle_mod, Lb):
    """The general kernels with their index checks on: no check fails and every output is the product build's, bit for bit."""
    from paper_2602_12011_gb300 import build as B
    th = _theta("lisa_and_long_arm")

    def outputs():
        _, gds, _ = _members(oracle_mod, Lb, "lisa_and_long_arm")
        out = []
        for flag in (0, Lb.PE_PREC_MIXED):
            r = Lb.loglike(gds, th, W.MODE_ALL | flag, dhhh=True)
            g = Lb.loglike_grad(gds, th, W.MODE_ALL | flag)
            out += [r["logl"], r["dhhh"], g["logl"], g["grad"]]
        out.append(Lb.fisher(gds, th, W.MODE_ALL))
        for gd in gds:
            gd.close()
        return out

    want = outputs()
    tl = Lb.load(B.build(variant="test"))
    prev = Lb.swap_library(tl)
    try:
        tl.pe_test_checked_take()
        got = outputs()
        assert tl.pe_test_checked_take() == 0
    finally:
        Lb.swap_library(prev)
    for a, b in zip(got, want):
        np.testing.assert_array_equal(a, b)
