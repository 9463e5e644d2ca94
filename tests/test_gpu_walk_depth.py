"""Stand-alone walks whose depth adapts to the walker's acceptance: the chain is that of the
one-step walk, bit for bit, in every precision, waveform and acceptance regime."""
import numpy as np
import pytest

from paper_2509_04336_gb300 import gwns, synth

from _util import event, priors

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def built():
    from paper_2509_04336_gb300 import build
    build.build()


def walk(w, ev, pri, precision, depth, live, u0, l0, star, steps, edges=None, noalloc=False):
    h = gwns.ns_init([gwns.make_config(w, pri, precision=precision, spec_depth=depth)], [ev])
    try:
        if edges is not None:
            gwns.ns_relbin_set(h, 0, edges, ev.theta_inj)
        n = u0.shape[0]
        out = [np.zeros_like(u0), np.zeros(n), np.zeros(n, np.int32), np.zeros(n, np.int32)]
        if noalloc:
            import torch
            t = lambda a: torch.tensor(a, device="cuda:0")
            dev = [t(a) for a in out]
            gwns.ns_walk_batch_noalloc(h, 0, t(live), t(u0), t(l0), star, steps, 2, 5, *dev)
            torch.cuda.synchronize()
            return [d.cpu().numpy() for d in dev]
        gwns.ns_walk_batch(h, 0, live, u0, l0, star, steps, 2, 5, *out)
        return out
    finally:
        gwns.ns_free(h)


@pytest.mark.parametrize("precision", [synth.PREC_FP64, synth.PREC_MIXED, synth.PREC_MIXED_FF])
@pytest.mark.parametrize("name,f_max,n", [("four_param_2det_taylorf2", 131.0, 7), ("bbh11_3det_4s_taylorf2", 128.0, 33),
                                          ("bbh11_3det_8s_phenomd", 400.0, 5)])
@pytest.mark.parametrize("quantile", [0.1, 0.5, 0.95])
def test_adaptive_depth_gives_the_one_step_chain(precision, name, f_max, n, quantile):
    # survivors across the prior, thresholds that accept most, half and hardly any of the moves
    w, ev = event(name, f_max=f_max)
    pri = priors(w, ev)
    u = synth.uniform_unit_cube(61, w.n_dim, 4)
    from oracle import prior as P
    th = np.stack([P.transform(x, pri) for x in u])
    h = gwns.ns_init([gwns.make_config(w, pri, precision=precision)], [ev])
    try:
        lnl = np.zeros(61)
        gwns.ns_likelihood_batch(h, 0, th, lnl)
    finally:
        gwns.ns_free(h)
    star = float(np.quantile(lnl, quantile))
    above = np.where(lnl > star)[0]
    pick = above[np.arange(n) % len(above)]
    u0, l0 = np.ascontiguousarray(u[pick]), np.ascontiguousarray(lnl[pick])
    args = (np.ascontiguousarray(u), u0, l0, star, 150)
    one = walk(w, ev, pri, precision, 1, *args)
    for kw in (dict(depth=0), dict(depth=0, noalloc=True)):
        got = walk(w, ev, pri, precision, kw.pop("depth"), *args, **kw)
        for a, b in zip(got, one):
            assert np.array_equal(a, b)
    assert one[2].sum() > 0 or quantile > 0.9
    if precision == synth.PREC_MIXED_FF:
        edges = gwns.ns_relbin_edges(ev.f_min, ev.df, ev.n_bins, 0.25)
        one, got = (walk(w, ev, pri, precision, d, *args, edges=edges) for d in (1, 0))
        for a, b in zip(got, one):
            assert np.array_equal(a, b)
