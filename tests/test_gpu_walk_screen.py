"""Walk steps whose proposal lies 1e-9 inside or outside a face of the cube, in one to four sampled
parameters: the FP32 screen keeps every step that the exact test keeps (one likelihood call), and
the exact test drops the others."""
from dataclasses import replace

import numpy as np
import pytest

from oracle import walk
from paper_2509_04336_gb300 import gwns, synth

from _util import event, priors

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def built():
    from paper_2509_04336_gb300 import build
    build.build()


@pytest.mark.parametrize("precision", [synth.PREC_FP64, synth.PREC_MIXED, synth.PREC_MIXED_FF])
@pytest.mark.parametrize("D", [1, 2, 3, 4])
def test_steps_at_the_faces_of_the_cube(precision, D):
    w, ev = event("four_param_2det_taylorf2", f_max=60.0)
    pri = priors(w, ev)
    pri = [p if i < D else replace(p, kind=synth.FIXED, value=float(ev.theta_inj[i])) for i, p in enumerate(pri)]
    n, n_s, it = 3000, 40, 2
    rng = np.random.default_rng(D)
    # two clumps in opposite corners: differences of up to the whole cube, where the scale's error counts
    surv = np.where(rng.random((n_s, 1)) < 0.5, 0.02, 0.98) + 0.02 * rng.uniform(-1, 1, (n_s, D))
    a, b, s = walk.de_step_draws(0, np.arange(n), it, n_s, D, (w.seed, 0))
    diff = s[:, None] * (surv[a] - surv[b])
    room = np.all(np.abs(diff) < 0.999, axis=1)
    assert room.sum() > 500
    u0 = np.where(room[:, None], np.clip(0.5 - 0.5 * diff, 0.0, 1.0), 0.5)   # start and proposal about the centre
    side = np.arange(n) % 4                                       # 1e-9 inside 1, inside 0, beyond 1, beyond 0
    x = np.array([1.0 - 1e-9, 1e-9, 1.0 + 1e-9, -1e-9])[side]
    d = np.arange(n) // 4 % D
    start = x - diff[np.arange(n), d]
    use = room & (start >= 0.0) & (start <= 1.0)
    u0[use, d[use]] = start[use]
    assert min(np.sum(use & (side == q)) for q in range(4)) > 50
    h = gwns.ns_init([gwns.make_config(w, pri, precision=precision)], [ev])
    try:
        out = [np.zeros((n, D)), np.zeros(n), np.zeros(n, np.int32), np.zeros(n, np.int32)]
        gwns.ns_walk_batch(h, 0, surv, u0, np.zeros(n), -1e300, 1, it, 0, *out)
    finally:
        gwns.ns_free(h)
    assert np.array_equal(out[3][use], (side[use] < 2).astype(np.int32))
