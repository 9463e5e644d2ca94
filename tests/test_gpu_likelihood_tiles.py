"""ns_likelihood_batch and ns_waveform at the edges of their tiles: a vector's result does not
depend on how many others share the call, its place in the tile or a non-finite neighbour."""
import numpy as np
import pytest

from oracle import likelihood as L
from paper_2509_04336_gb300 import gwns, synth

from _util import event, priors, prior_draws

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def built():
    from paper_2509_04336_gb300 import build
    build.build()


# 304 vectors a tile of one, then two, three, ... up to sixteen (TaylorF2) and four (IMRPhenomD form)
@pytest.mark.parametrize("precision", [synth.PREC_FP64, synth.PREC_MIXED, synth.PREC_MIXED_FF])
@pytest.mark.parametrize("name,sizes", [("four_param_2det_taylorf2", (1, 304, 305, 911, 1217, 4861, 4900)),
                                        ("bbh11_3det_8s_phenomd", (1, 305, 913, 1300))])
def test_a_vector_alone_and_in_any_tile(precision, name, sizes):
    w, ev = event(name, f_max=180.0)
    _, th = prior_draws(w, ev, 40, 3)
    h = gwns.ns_init([gwns.make_config(w, priors(w, ev), precision=precision)], [ev])
    try:
        one = np.zeros(40)
        for i in range(40):
            gwns.ns_likelihood_batch(h, 0, np.ascontiguousarray(th[i:i + 1]), one[i:i + 1])
        for n in sizes:
            got = np.zeros(n)
            gwns.ns_likelihood_batch(h, 0, np.ascontiguousarray(th[np.arange(n) % 40]), got)
            # the whole CTA and a lone warp sum a proposal in one order, so the bits agree
            assert np.array_equal(got, one[np.arange(n) % 40]), n
        import torch
        n = sizes[-1]
        many = th[np.arange(n) % 40].copy()
        many[5, 3], many[n - 1, 0] = np.nan, -1.0
        dev, out = torch.tensor(many, device="cuda:0"), torch.zeros(n, device="cuda:0", dtype=torch.float64)
        gwns.ns_likelihood_batch(h, 0, dev, out)
        got, bad = out.cpu().numpy(), np.array([5, n - 1])
        assert np.all(np.isnan(got[bad]))
        good = np.setdiff1d(np.arange(n), bad)
        assert np.array_equal(got[good], one[good % 40])
    finally:
        gwns.ns_free(h)


@pytest.mark.parametrize("name,f_max", [("four_param_2det_taylorf2", 51.75), ("bbh11_3det_4s_taylorf2", 512.0),
                                        ("bbh11_3det_8s_phenomd", 1500.25)])
@pytest.mark.parametrize("n", [1, 3, 700])
def test_waveform_spans(name, f_max, n):
    # 128-bin rows in spans of one row up to the whole grid; FP64 against the oracle: both sides
    # carry phases of ~1e3 cycles to ~1e-13 cycles, so 1e-10 of the largest strain is ample
    w, ev = event(name, f_max=f_max)
    _, th = prior_draws(w, ev, 3, 8)
    h = gwns.ns_init([gwns.make_config(w, priors(w, ev))], [ev])
    try:
        big = np.ascontiguousarray(th[np.arange(n) % 3])
        re, im = (np.zeros((n, len(ev.detectors), ev.n_bins)) for _ in range(2))
        gwns.ns_waveform(h, 0, big, re, im)
    finally:
        gwns.ns_free(h)
    for i in {0, n // 2, n - 1}:
        for d in range(len(ev.detectors)):
            want = L.project(ev, d, big[i], w.waveform)
            assert np.max(np.abs(re[i, d] + 1j * im[i, d] - want)) <= 1e-10 * np.max(np.abs(want))


@pytest.mark.parametrize("name,sizes", [("bbh11_3det_4s_taylorf2", (1, 305, 911, 4900)),
                                        ("bbh11_3det_8s_phenomd", (1, 305, 1300))])
def test_relative_binning_alone_and_in_any_tile(name, sizes):
    # a warp takes every fourth vector of the tile: the same operations as for a vector alone
    w, ev = event(name, f_max=180.0)
    _, th = prior_draws(w, ev, 40, 3)
    h = gwns.ns_init([gwns.make_config(w, priors(w, ev), precision=synth.PREC_MIXED_FF)], [ev])
    try:
        gwns.ns_relbin_set(h, 0, gwns.ns_relbin_edges(ev.f_min, ev.df, ev.n_bins, 0.25), ev.theta_inj)
        one = np.zeros(40)
        for i in range(40):
            gwns.ns_likelihood_batch(h, 0, np.ascontiguousarray(th[i:i + 1]), one[i:i + 1])
        assert np.all(np.isfinite(one))
        import torch
        for n in sizes:
            many = th[np.arange(n) % 40].copy()
            bad = np.unique([n // 3, n - 1]) if n > 1 else np.array([], int)
            many[bad, 3] = np.nan
            dev, out = torch.tensor(many, device="cuda:0"), torch.zeros(n, device="cuda:0", dtype=torch.float64)
            gwns.ns_likelihood_batch(h, 0, dev, out)
            got = out.cpu().numpy()
            good = np.setdiff1d(np.arange(n), bad)
            assert np.all(np.isnan(got[bad])) and np.array_equal(got[good], one[good % 40]), n
    finally:
        gwns.ns_free(h)


@pytest.mark.parametrize("precision,relbin", [(synth.PREC_FP64, False), (synth.PREC_MIXED, False),
                                              (synth.PREC_MIXED_FF, False), (synth.PREC_MIXED_FF, True)])
@pytest.mark.parametrize("name", ["four_param_2det_taylorf2", "bbh11_3det_8s_phenomd"])
@pytest.mark.parametrize("n_live", [300, 305, 911, 1217])
def test_initial_live_points_in_any_tile(precision, relbin, name, n_live):
    # the live points' ln L, formed from the unit cube in tiles of one to five, against the same
    # points' physical vectors.  The posterior of a run of no batches weighs them by ln L alone.
    # Tolerance: each side's own bound, 1e-11 (FP64) or 1e-6 of max(|ln L|, SNR^2 / 2)
    w, ev = event(name, f_max=120.0, n_live=n_live)
    h = gwns.ns_init([gwns.make_config(w, priors(w, ev), precision=precision)], [ev])
    try:
        if relbin:
            gwns.ns_relbin_set(h, 0, gwns.ns_relbin_edges(ev.f_min, ev.df, ev.n_bins, 0.25), ev.theta_inj)
        theta, logw = gwns.ns_posterior(h, 0)
        assert theta.shape == (n_live, 11)
        lnl = np.zeros(n_live)
        gwns.ns_likelihood_batch(h, 0, np.ascontiguousarray(theta), lnl)
    finally:
        gwns.ns_free(h)
    top = np.argmax(lnl)
    tol = (1e-11 if precision == synth.PREC_FP64 else 1e-6) * np.maximum(np.abs(lnl), 0.5 * w.snr ** 2)
    assert np.all(np.abs((logw - logw[top]) - (lnl - lnl[top])) <= 2 * (tol + tol[top]))
