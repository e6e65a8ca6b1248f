"""GPU tests of the per-sample preparation, the work-list scan and the last reduction across the rules that pick
their forms: eight threads or one to a sample (8,192 samples), one thread or a run of pairs per scan thread
(1,024 pairs), one warp or one CTA per sample in the reductions (64 tiles of a grid).

Every form has to give a sample the same bits, so the values are compared exactly with the sample alone.
"""
import numpy as np
import pytest

from paper_2602_12011_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def Lb():
    from paper_2602_12011_gb300 import _lib
    _lib.lib()
    return _lib


def _det(Lb, T, cfg=W.LISA):
    d = Lb.Detector(cfg, T, *W.grid(T))
    d.inject(W.theta_injection(T), W.MODE_ALL, W.normals(d.nb, 3))
    return d


@pytest.mark.parametrize("B", [1, 7, 31, 33, 1023, 1025, 8191, 8193])
def test_batch_sizes_give_a_sample_the_same_bits(Lb, B):
    T = 2.0 ** 13
    d = [_det(Lb, T), _det(Lb, T, W.TIANQIN)]
    th = W.draw_prior(B, 41, T)
    th[B // 2, 1] = 1.0                                  # equal masses: the odd modes vanish
    th[B // 3, 2] = 1.0                                  # out of domain
    for flag in (0, Lb.PE_PREC_MIXED):
        r = Lb.loglike(d, th, W.MODE_ALL | flag, dhhh=True, status=True)
        g = Lb.loglike_grad(d, th, W.MODE_ALL | flag)
        for s in sorted({0, B // 3, B // 2, B - 1}):
            one = Lb.loglike(d, th[s:s + 1], W.MODE_ALL | flag, dhhh=True, status=True)
            assert one["logl"][0] == r["logl"][s] and one["status"][0] == r["status"][s]
            assert np.array_equal(one["dhhh"][0], r["dhhh"][s])
            og = Lb.loglike_grad(d, th[s:s + 1], W.MODE_ALL | flag)
            assert np.array_equal(og["grad"][0], g["grad"][s]) and og["logl"][0] == g["logl"][s]


@pytest.mark.parametrize("tiles", [64, 65])
def test_reductions_at_the_rule_between_warp_and_cta(Lb, tiles):
    """<d|h> and <h|h> against sums over the library's own per-bin signal, on either side of the rule: FP64 sums
    of up to 8,320 terms in another order, each term formed with a few more roundings (1e-12 of the sums of
    magnitudes, about 8,320 x 2^-53)."""
    T, nb = 2.0 ** 18, tiles * 128
    d = Lb.Detector(W.LISA, T, 27, nb)
    th = W.theta_injection(T)
    th[0] = 2e5
    d.inject(th, W.MODE_ALL, W.normals(nb, 5))
    rng = np.random.Generator(np.random.PCG64(5))
    data = d.signal(th, W.MODE_ALL) + rng.standard_normal((3, nb)) * np.sqrt(d.psd() * T / 4.0)
    d.set_data(data)
    t2 = th.copy()
    t2[6] += 0.3
    h, w = d.signal(t2, W.MODE_ALL), 4.0 / (d.psd() * T)
    r = Lb.loglike([d], t2, W.MODE_ALL, dhhh=True)
    dh, hh = w * (data.conj() * h).real, w * np.abs(h) ** 2
    assert np.all(np.abs(r["dhhh"][0, 0, :, 0] - dh.sum(1)) <= 1e-12 * np.abs(dh).sum(1))
    assert np.all(np.abs(r["dhhh"][0, 0, :, 1] - hh.sum(1)) <= 1e-12 * hh.sum(1))
    g = Lb.loglike_grad([d], t2, W.MODE_ALL)
    scale = 0.5 * d.data_norm().sum() + abs(dh.sum()) + hh.sum()
    assert abs(g["logl"][0] - r["logl"][0]) <= 1e-12 * scale


@pytest.mark.parametrize("B", [6143, 6144, 6145])
def test_batches_at_the_rule_between_eight_threads_and_one(Lb, B):
    test_batch_sizes_give_a_sample_the_same_bits(Lb, B)
