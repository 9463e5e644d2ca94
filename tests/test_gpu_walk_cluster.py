"""FP64 and FP64-phase walks of few walkers, each on a cluster of CTAs: a walker's chain is the same
whatever the size of its launch (four, two or one CTA a walker)."""
import numpy as np
import pytest

from paper_2509_04336_gb300 import gwns, synth

from _util import event, priors, prior_draws

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def built():
    from paper_2509_04336_gb300 import build
    build.build()


@pytest.mark.parametrize("precision", [synth.PREC_FP64, synth.PREC_MIXED])
@pytest.mark.parametrize("name,f_max", [("four_param_2det_taylorf2", 200.0), ("bbh11_3det_8s_phenomd", 250.0)])
@pytest.mark.parametrize("depth", [0, 1, 8])
def test_chain_does_not_depend_on_the_launch(precision, name, f_max, depth):
    w, ev = event(name, f_max=f_max)
    pri = priors(w, ev)
    u, th = prior_draws(w, ev, 80, 6)
    h = gwns.ns_init([gwns.make_config(w, pri, precision=precision, spec_depth=depth)], [ev])
    try:
        lnl = np.zeros(80)
        gwns.ns_likelihood_batch(h, 0, th, lnl)
        star = float(np.median(lnl))
        above = np.where(lnl > star)[0]
        u0, l0 = np.ascontiguousarray(u[above]), np.ascontiguousarray(lnl[above])
        pick = np.arange(160) % len(above)

        def walk(n):   # walkers 0 .. n-1
            out = [np.zeros((n, w.n_dim)), np.zeros(n), np.zeros(n, np.int32), np.zeros(n, np.int32)]
            gwns.ns_walk_batch(h, 0, np.ascontiguousarray(u), np.ascontiguousarray(u0[pick[:n]]),
                               np.ascontiguousarray(l0[pick[:n]]), star, 40, 1, 0, *out)
            return out

        full = walk(160)                     # more walkers than SMs: one CTA each
        for n in (1, 38, 39, 76, 77):        # 4 CTAs a walker up to 38 walkers (152 SMs), 2 up to 76
            for a, b in zip(walk(n), full):
                assert np.array_equal(a, b[:n]), n
        # the abort flag ends the walks of every rank after their first round, above L*
        gwns.ns_set_abort(h, True)
        with pytest.raises(gwns.GwnsError) as e:
            walk(20)
        assert e.value.code == gwns.NS_ETIMEOUT
        gwns.ns_set_abort(h, False)
        for a, b in zip(walk(20), full):
            assert np.array_equal(a, b[:20])
    finally:
        gwns.ns_free(h)


@pytest.mark.parametrize("precision", [synth.PREC_FP64, synth.PREC_MIXED])
def test_walks_of_one_round(precision):
    # one or two steps: a walk's first round is its last, so what the ranks exchange in it is all
    w, ev = event("four_param_2det_taylorf2", f_max=60.0)
    u, th = prior_draws(w, ev, 90, 8)
    h = gwns.ns_init([gwns.make_config(w, priors(w, ev), precision=precision, spec_depth=8)], [ev])
    try:
        lnl = np.zeros(90)
        gwns.ns_likelihood_batch(h, 0, th, lnl)
        star = float(np.quantile(lnl, 0.1))
        above = np.where(lnl > star)[0]
        pick = above[np.arange(160) % len(above)]
        for steps in (1, 2):
            def walk(n):
                out = [np.zeros((n, w.n_dim)), np.zeros(n), np.zeros(n, np.int32), np.zeros(n, np.int32)]
                gwns.ns_walk_batch(h, 0, np.ascontiguousarray(u), np.ascontiguousarray(u[pick[:n]]),
                                   np.ascontiguousarray(lnl[pick[:n]]), star, steps, 1, 0, *out)
                return out

            full = walk(160)
            assert full[3].sum() > 0
            for n in (1, 38, 76):
                for a, b in zip(walk(n), full):
                    assert np.array_equal(a, b[:n]), n
    finally:
        gwns.ns_free(h)
