"""Walks whose differences come from an array far larger than a live set: the handle's scratch does not
grow with it, and the chain is that of the walk that allocates nothing."""
import numpy as np
import pytest

from paper_2509_04336_gb300 import gwns, synth

from _util import event, priors

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def built():
    from paper_2509_04336_gb300 import build
    build.build()


@pytest.mark.parametrize("precision", [synth.PREC_FP64, synth.PREC_MIXED, synth.PREC_MIXED_FF])
def test_large_survivor_array(precision):
    import torch
    w, ev = event("four_param_2det_taylorf2", f_max=60.0)
    n, big = 40, 1 << 22                       # 4.2 M points of 4 coordinates: 134 MB
    u0 = synth.uniform_unit_cube(n, w.n_dim, 3)
    live = torch.rand((big, w.n_dim), dtype=torch.float64, device="cuda:0", generator=torch.Generator("cuda:0").manual_seed(4))
    dev = lambda a: torch.tensor(a, device="cuda:0")
    h = gwns.ns_init([gwns.make_config(w, priors(w, ev), precision=precision)], [ev])
    try:
        def walk(surv):
            out = [dev(a) for a in (np.zeros_like(u0), np.zeros(n), np.zeros(n, np.int32), np.zeros(n, np.int32))]
            gwns.ns_walk_batch(h, 0, surv, dev(u0), dev(np.zeros(n)), -1e300, 60, 2, 5, *out)
            torch.cuda.synchronize()
            return [a.cpu().numpy() for a in out]

        walk(live[:1000])
        free = torch.cuda.mem_get_info()[0]
        got = walk(live)
        assert free - torch.cuda.mem_get_info()[0] < 16 << 20
        out = [dev(a) for a in (np.zeros_like(u0), np.zeros(n), np.zeros(n, np.int32), np.zeros(n, np.int32))]
        gwns.ns_walk_batch_noalloc(h, 0, live, dev(u0), dev(np.zeros(n)), -1e300, 60, 2, 5, *out)   # never pairs
        torch.cuda.synchronize()
        for a, b in zip(got, out):
            assert np.array_equal(a, b.cpu().numpy())
        assert got[2].sum() > 0
    finally:
        gwns.ns_free(h)
