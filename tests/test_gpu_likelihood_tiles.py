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
