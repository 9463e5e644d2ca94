"""The sampler's first speculation cap follows what a speculative proposal costs: the largest where
rounds are dominated by fixed costs or end at their first acceptance, a small one where every
proposal of a round is evaluated over a thousand bins or more."""
import pytest

from paper_2509_04336_gb300 import gwns, synth

from _util import event, priors

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def built():
    from paper_2509_04336_gb300 import build
    build.build()


@pytest.mark.parametrize("precision,eps,cap", [
    (synth.PREC_MIXED_FF, None, 32),     # rounds end at their first acceptance
    (synth.PREC_MIXED_FF, 0.25, 32),     # ~120 coarse bins
    (synth.PREC_MIXED_FF, 1e-3, 4),      # ~3,900 coarse bins, a warp per proposal
    (synth.PREC_MIXED, None, 4),
])
def test_first_cap(precision, eps, cap):
    w, ev = event("bbh11_3det_8s_phenomd", f_max=512.0, n_live=40)
    h = gwns.ns_init([gwns.make_config(w, priors(w, ev), precision=precision)], [ev])
    try:
        if eps is not None:
            edges = gwns.ns_relbin_edges(ev.f_min, ev.df, ev.n_bins, eps)
            assert (len(edges) > 2500) == (cap == 4)
            gwns.ns_relbin_set(h, 0, edges, ev.theta_inj)
        gwns.ns_step(h, 1, 1)
        _, prog = gwns.ns_step(h, 1, 1)
        assert prog[0]["spec_cap"] == cap
    finally:
        gwns.ns_free(h)
