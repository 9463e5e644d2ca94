"""What is measured: the calls that a user of the sampler makes, from one likelihood to whole runs.

Kinds of case, each through the public binding (paper_2509_04336_gb300.gwns):
  lnl    ns_likelihood_batch on device tensors: half prior draws (as an initial live set), half
         points around the injection (as posterior points evaluated again)
  wave   ns_waveform on device tensors: detector strains of n parameter vectors
  walk   ns_walk_batch on device tensors: one batch of constrained differential-evolution walks
         of half the live points, part-way through a run ("spread" is the width of the live set in
         the unit cube, 1 the prior); "relbin" > 0: on the relative-binning likelihood
  flow   ns_flow_train: one retraining of the flow proposal on host points (training state set
         back to the same weights first)
  run    a whole program: ns_init from host data, ns_step, ns_evidence, ns_posterior, ns_free;
         "batches" 0 means to the stopping rule
A case names a workload of synth.workload; f_max, n_live and the precision (0 FP64, 1 FP32 sums
with the FP64 phase, 2 FP32 sums with the float-float phase) vary.

exact() is a plain restatement of the model in 64-bit torch and numpy.
"""
import math
from dataclasses import replace

import numpy as np
import torch

from paper_2509_04336_gb300 import gwns, synth

DEV = "cuda:0"
W4P, W4S, W8S, W8F = ("four_param_2det_taylorf2", "bbh11_3det_4s_taylorf2", "bbh11_3det_8s_phenomd",
                      "bbh11_3det_8s_phenomd_flow")
F_MAX = {W4P: 512.0, W4S: 1024.0, W8S: 2048.0, W8F: 2048.0}


def listed():
    return [
        # the smallest call: one likelihood from a program of the user's own (an optimiser, a check)
        dict(name="lnl_one_4p_fp64", kind="lnl", w=W4P, f_max=512.0, prec=0, n=1),
        # the initial live set of the 11-parameter event, in its configured precision
        dict(name="lnl_4s_mixed", kind="lnl", w=W4S, f_max=1024.0, prec=1, n=1000),
        # a large posterior evaluated again on the 16,225-bin event
        dict(name="lnl_8s_ff", kind="lnl", w=W8S, f_max=2048.0, prec=2, n=4001),
        # strains of posterior points, as a reconstruction plot or an injection set needs them
        dict(name="wave_8s", kind="wave", w=W8S, f_max=2048.0, prec=2, n=33),
        # one batch of the small FP64 event: 50 walkers, launch and latency count
        dict(name="walk_4p_fp64", kind="walk", w=W4P, f_max=512.0, prec=0, n_live=100, steps=80, spread=0.5, relbin=0.0),
        # one batch of the 11-parameter event: 500 walkers, in the fast precision and the configured one
        dict(name="walk_4s_ff", kind="walk", w=W4S, f_max=1024.0, prec=2, n_live=1000, steps=600, spread=0.3, relbin=0.0),
        dict(name="walk_4s_mixed", kind="walk", w=W4S, f_max=1024.0, prec=1, n_live=1000, steps=240, spread=0.3, relbin=0.0),
        # one batch of the long IMRPhenomD-form event: 1000 walkers over thousands of bins
        dict(name="walk_8s_ff", kind="walk", w=W8S, f_max=2048.0, prec=2, n_live=2000, steps=240, spread=0.3, relbin=0.0),
        # the same on the compressed likelihood
        dict(name="walk_8s_relbin", kind="walk", w=W8S, f_max=2048.0, prec=2, n_live=2000, steps=240, spread=0.3, relbin=0.25),
        # one retraining of the flow proposal: 2000 survivors, 50 epochs
        dict(name="flow_train_8s", kind="flow", w=W8F, f_max=64.0, prec=2, n=2000, epochs=50, layers=8),
        # the small event from its data to its evidence and posterior
        dict(name="run_4p_fp64", kind="run", w=W4P, f_max=512.0, prec=0, n_live=100, batches=0, events=1),
        # the first batches of the 11-parameter event, start-up and read-out included
        dict(name="run_4s_ff", kind="run", w=W4S, f_max=1024.0, prec=2, n_live=1000, batches=10, events=1),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["lnl", "lnl", "wave", "walk", "walk", "walk", "flow", "run"])
    w = rng.choice([W4P, W4S, W8S])
    c = dict(kind=kind, w=w, f_max=round(rng.uniform(0.25, 1.0) * F_MAX[w], 3), prec=rng.randrange(3))
    # bins of an evaluation relative to the 16,225 of the longest, and the cost of a precision
    cost = (c["f_max"] / F_MAX[w]) * {W4P: 0.02, W4S: 0.03, W8S: 1.0}[w] * (30.0, 6.0, 1.0)[c["prec"]]
    if kind == "lnl":
        c["n"] = _log_int(rng, 1, max(1, min(4000, int(4000 / cost))))
    elif kind == "wave":
        c["n"] = _log_int(rng, 1, 33)
    elif kind == "walk":
        c["n_live"] = _log_int(rng, 20, max(21, min(2000, int(1600 / cost))))
        c["steps"] = _log_int(rng, 10, max(11, min(400, int(400000 / (cost * c["n_live"])))))
        c["spread"] = round(rng.uniform(0.2, 1.0), 3)
        c["relbin"] = 0.25 if c["prec"] == 2 and rng.random() < 0.25 else 0.0
    elif kind == "flow":
        c.update(w=W8F, f_max=64.0, prec=2, n=_log_int(rng, 50, 2000), epochs=rng.randint(1, 50), layers=rng.randint(1, 8))
    else:
        c.update(w=rng.choice([W4P, W4S]), prec=rng.choice([0, 2]), n_live=_log_int(rng, 50, 500),
                 batches=rng.randint(1, 6), events=rng.randint(1, 3))
        c["f_max"] = round(rng.uniform(0.25, 1.0) * F_MAX[c["w"]], 3)
    return c


# ------------------------------------------------------------------ the model, in plain 64 bits
G_SUN = 1.32712440018e20
C_LIGHT = 299792458.0
MSUN_S = G_SUN / C_LIGHT ** 3
MPC = 3.085677581491367e22
X_INS, X_AMP, X_CUT = 0.018, 0.014, 0.2
S2, S3, S4, B2, B3 = 50.0, -100.0, 40.0, 1.0, 1.0e-5
A2_, A3_, A4_, A5_ = 0.01, 0.5, 0.05, 1.0
G1, G2, G3 = 0.006, 0.9, 1.3


def _pn(eta, delta, c1, c2):
    s, a, pi = 0.5 * (c1 + c2), 0.5 * (c1 - c2), math.pi
    z = torch.zeros_like(eta)
    p5 = (38645 * pi / 756 - 65 * pi * eta / 9 - (732985 / 2268 - 24260 * eta / 81 - 340 * eta ** 2 / 9) * s
          - (732985 / 2268 + 140 * eta / 9) * delta * a)
    p = [z + 1, z, 3715 / 756 + 55 * eta / 9,
         -16 * pi + 113 / 3 * delta * a + (113 / 3 - 76 * eta / 3) * s,
         15293365 / 508032 + 27145 * eta / 504 + 3085 * eta ** 2 / 72 + (-405 / 8 + 200 * eta) * a ** 2
         - 405 / 4 * delta * a * s + (-405 / 8 + 5 * eta / 2) * s ** 2,
         p5,
         11583231236531 / 4694215680 - 6848 * 0.5772156649015329 / 21 - 640 * pi ** 2 / 3
         + (-15737765635 / 3048192 + 2255 * pi ** 2 / 12) * eta + 76055 * eta ** 2 / 1728 - 127825 * eta ** 3 / 1296
         - 6848 / 21 * math.log(4.0) + 2270 * pi / 3 * delta * a + (2270 * pi / 3 - 520 * pi * eta) * s,
         77096675 * pi / 254016 + 378515 * pi * eta / 1512 - 74045 * pi * eta ** 2 / 756
         + (-25150083775 / 3048192 + 10566655595 * eta / 762048 - 1042165 * eta ** 2 / 3024 + 5345 * eta ** 3 / 36) * s
         + (-25150083775 / 3048192 + 26804935 * eta / 6048 - 1985 * eta ** 2 / 48) * delta * a]
    return p, {5: 3 * p5, 6: z - 6848 / 21}


def _tf2(x, eta, p, pl):
    """TaylorF2 phase at x = M f, and its slope."""
    v = (math.pi * x) ** (1 / 3)
    lv = torch.log(v)
    s, ds = torch.zeros_like(v), torch.zeros_like(v)
    for k in range(8):
        t = p[k] + (pl[k] * lv if k in pl else 0.0)
        s = s + t * v ** (k - 5)
        ds = ds + v ** (k - 5) * ((k - 5) * t + (pl[k] if k in pl else 0.0)) / (3 * x)
    return 3 / (128 * eta) * s, 3 / (128 * eta) * ds


def _phase_amp(th, f, wf, cut):
    """(phase without t_c and phi_c, amplitude shape, mask of the bins below the cutoff), [n][bins]."""
    q, c1, c2 = th[:, 1:2], th[:, 2:3], th[:, 3:4]
    eta, delta = q / (1 + q) ** 2, (1 - q) / (1 + q)
    M = th[:, 0:1] * eta ** -0.6 * MSUN_S
    x = M * f[None, :]
    p, pl = _pn(eta, delta, c1, c2)
    if wf == synth.TAYLORF2:
        return _tf2(x, eta, p, pl)[0], torch.ones_like(x), (f[None, :] <= 1 / (6 ** 1.5 * math.pi * M)) | (not cut)
    at = (c1 + c2 * q ** 2) / (1 + q ** 2)
    af = at + at * eta * (-0.1229 * at + 0.4537 * eta - 2.8904) + eta * (2 * 3 ** 0.5 - 3.5171 * eta + 2.5763 * eta ** 2)
    om, qf = 1.5251 - 1.1568 * (1 - af) ** 0.1292, 0.7 + 1.4187 * (1 - af) ** -0.4990
    fr = om / (2 * math.pi * (1 - (0.0572 * eta + 0.498 * eta ** 2)))
    fd = fr / (2 * qf)

    def ins(x):
        s, ds = _tf2(x, eta, p, pl)
        return (s + (0.75 * S2 * x ** (4 / 3) + 0.6 * S3 * x ** (5 / 3) + 0.5 * S4 * x ** 2) / eta,
                ds + (S2 * x ** (1 / 3) + S3 * x ** (2 / 3) + S4 * x) / eta)

    x1, x2 = X_INS + torch.zeros_like(eta), 0.5 * fr
    p1, d1 = ins(x1)
    b1 = eta * d1 - B2 / x1 - B3 / x1 ** 4
    b0 = eta * p1 - b1 * x1 - B2 * torch.log(x1) + B3 / (3 * x1 ** 3)
    p2 = (b0 + b1 * x2 + B2 * torch.log(x2) - B3 / (3 * x2 ** 3)) / eta
    d2 = (b1 + B2 / x2 + B3 / x2 ** 4) / eta
    lor = A4_ * torch.atan((x2 - A5_ * fr) / fd)
    dlor = A4_ * fd / ((x2 - A5_ * fr) ** 2 + fd ** 2)
    a1 = eta * d2 - A2_ / x2 ** 2 - A3_ * x2 ** -0.25 - dlor
    a0 = eta * p2 - a1 * x2 + A2_ / x2 - 4 / 3 * A3_ * x2 ** 0.75 - lor
    psi = torch.where(x < x1, ins(x)[0], torch.where(
        x < x2, (b0 + b1 * x + B2 * torch.log(x) - B3 / (3 * x ** 3)) / eta,
        (a0 + a1 * x - A2_ / x + 4 / 3 * A3_ * x ** 0.75 + A4_ * torch.atan((x - A5_ * fr) / fd)) / eta))
    s, a = 0.5 * (c1 + c2), 0.5 * (c1 - c2)
    k2, k3 = -323 / 224 + 451 * eta / 168, 27 * delta * a / 8 + (27 / 8 - 11 * eta / 6) * s
    gd = G3 * fd
    xp = torch.abs(fr + gd * (math.sqrt(1 - G2 ** 2) - 1) / G2)

    def inner_amp(x):
        v = (math.pi * x) ** (1 / 3)
        return 1 + k2 * v ** 2 + k3 * v ** 3, (2 * k2 * v + 3 * k3 * v ** 2) * v / (3 * x)

    def ring_amp(x):
        den = (x - fr) ** 2 + gd ** 2
        r = G1 * gd / den * torch.exp(-G2 * (x - fr) / gd)
        return r, r * (-2 * (x - fr) / den - G2 / gd)

    (y0, e0), (y1, e1) = inner_amp(X_AMP + torch.zeros_like(eta)), ring_amp(xp)
    span = xp - X_AMP
    t = (x - X_AMP) / span
    mid = ((2 * t ** 3 - 3 * t ** 2 + 1) * y0 + (t ** 3 - 2 * t ** 2 + t) * span * e0 + (3 * t ** 2 - 2 * t ** 3) * y1
           + (t ** 3 - t ** 2) * span * e1)
    amp = torch.where(x < X_AMP, inner_amp(x)[0], torch.where(x < xp, mid, ring_amp(x)[0]))
    return psi, amp, (x <= X_CUT) | (not cut)


def _strain(geo, th, f, wf, cut=True):
    """Detector strains [n][det][bins] of th [n][11]; geo = (vertex, x arm, y arm) [det][3], gmst."""
    vert, xa, ya, gmst = geo
    psi, shape, on = _phase_amp(th, f, wf, cut)
    mcs = th[:, 0] * MSUN_S
    amp = math.sqrt(5 / 24) * math.pi ** (-2 / 3) * mcs ** (5 / 6) / (th[:, 4] * MPC / C_LIGHT)
    ph = th[:, 9] - gmst
    ct, st = torch.sin(th[:, 10]), torch.cos(th[:, 10])
    sp, cp, ss, cs = torch.sin(ph), torch.cos(ph), torch.sin(th[:, 6]), torch.cos(th[:, 6])
    X = torch.stack([sp * cs - ss * cp * ct, -(cp * cs + ss * sp * ct), ss * st], 1)
    Y = torch.stack([-sp * ss - cs * cp * ct, cp * ss - cs * sp * ct, st * cs], 1)
    N = torch.stack([st * cp, st * sp, ct], 1)
    xX, xY, yX, yY = X @ xa.T, Y @ xa.T, X @ ya.T, Y @ ya.T          # [n][det]
    fp, fc = 0.5 * (xX ** 2 - xY ** 2 - yX ** 2 + yY ** 2), xX * xY - yX * yY
    dt = -(N @ vert.T) / C_LIGHT
    ci = torch.cos(th[:, 5:6])
    pol = torch.complex(fp * 0.5 * (1 + ci ** 2), -fc * ci) * amp[:, None]
    turns = (psi - 2 * th[:, 7:8] - math.pi / 4)[:, None, :] / (2 * math.pi) + (th[:, 8:9] + dt)[:, :, None] * f
    turns = 2 * math.pi * (turns - torch.round(turns))
    env = (f ** (-7 / 6) * shape * on)[:, None, :]
    return pol[:, :, None] * torch.complex(env * torch.cos(turns), -env * torch.sin(turns))


def _torch_event(ev):
    t = lambda x: torch.tensor(np.array(x), dtype=torch.float64, device=DEV)  # noqa: E731
    geo = (t([d.vertex for d in ev.detectors]), t([d.x_arm for d in ev.detectors]), t([d.y_arm for d in ev.detectors]), ev.gmst)
    data = torch.tensor(np.array([d.data for d in ev.detectors]), device=DEV)
    wt = 4 * ev.df / t([d.psd for d in ev.detectors])
    return geo, t(synth.frequencies(ev.f_min, ev.df, ev.n_bins)), data, wt


class _Exact:
    """ln L of theta [n][11] in 64 bits; edges and theta0: the relative-binning likelihood."""

    def __init__(self, ev, wf, edges=None):
        self.wf, self.ev, self.edges = wf, ev, edges
        self.geo, self.f, self.d, self.wt = _torch_event(ev)
        self.dd = (self.d.abs() ** 2 * self.wt).sum()
        if edges is not None:
            th0 = torch.tensor(ev.theta_inj, dtype=torch.float64, device=DEV)[None]
            self.E = torch.tensor(np.asarray(edges, dtype=np.int64), device=DEV)
            self.fe = ev.f_min + ev.df * self.E.double()
            self.h0e = _strain(self.geo, th0, self.fe, wf, False)[0]
            h0 = _strain(self.geo, th0, self.f, wf, False)[0]
            b = torch.bucketize(torch.arange(ev.n_bins, device=DEV), self.E, right=True) - 1
            x = self.f - self.fe[b]
            nb, nd = len(edges) - 1, len(ev.detectors)
            zero = torch.zeros(nd, nb, dtype=torch.float64, device=DEV)
            add = lambda v: (torch.complex(zero, zero) if v.is_complex() else zero).index_add(1, b, v)  # noqa: E731
            cd, pw = self.d.conj() * h0 * self.wt, h0.abs() ** 2 * self.wt
            self.A, self.B = (add(cd), add(cd * x)), (add(pw), add(pw * x), add(pw * x * x))

    def __call__(self, th, rows=None):
        rows = rows or max(1, int(6e6) // (self.f.numel() * self.d.shape[0]))
        return torch.cat([self._some(th[i:i + rows]) for i in range(0, th.shape[0], rows)])

    def _some(self, th):
        h = _strain(self.geo, th, self.f, self.wf)
        dh, hh = (self.d.conj() * h).real * self.wt, (h.real ** 2 + h.imag ** 2) * self.wt
        if self.edges is None:
            return -0.5 * (self.dd - 2 * dh.sum((1, 2)) + hh.sum((1, 2)))
        k_end = (h[:, 0].abs() > 0).sum(1)
        full = (self.E[None, 1:] <= k_end[:, None]) & (self.E[None, 1:] < self.ev.n_bins)
        lo = self.E[full.sum(1)]
        tail = (torch.arange(self.f.numel(), device=DEV)[None, :] >= lo[:, None])[:, None, :]
        r = _strain(self.geo, th, self.fe, self.wf, False) / self.h0e
        r0, r1 = r[:, :, :-1], (r[:, :, 1:] - r[:, :, :-1]) / (self.fe[1:] - self.fe[:-1])
        on = full[:, None, :]
        cdh = (self.A[0] * r0 + self.A[1] * r1).real * on
        chh = (self.B[0] * r0.abs() ** 2 + 2 * self.B[1] * (r0.conj() * r1).real + self.B[2] * r1.abs() ** 2) * on
        return -0.5 * (self.dd - 2 * (cdh.sum((1, 2)) + (dh * tail).sum((1, 2))) + chh.sum((1, 2)) + (hh * tail).sum((1, 2)))


def _theta(pri, u):
    """Physical parameters [n][11] of unit-cube points u [n][D] (torch)."""
    out, d = [], 0
    for p in pri:
        if p.kind == synth.FIXED:
            out.append(torch.full_like(u[:, 0], p.value))
            continue
        v = u[:, d]
        d += 1
        if p.kind == synth.UNIFORM:
            out.append(p.lo + v * (p.hi - p.lo))
        elif p.kind == synth.POWERLAW:
            e = p.alpha + 1
            out.append((p.lo ** e + v * (p.hi ** e - p.lo ** e)) ** (1 / e))
        elif p.kind == synth.SINE:
            out.append(torch.acos((math.cos(p.lo) - v * (math.cos(p.lo) - math.cos(p.hi))).clamp(-1, 1)))
        else:
            out.append(torch.asin((math.sin(p.lo) + v * (math.sin(p.hi) - math.sin(p.lo))).clamp(-1, 1)))
    return torch.stack(out, 1)


def _unit(pri, th):
    """The unit-cube point of one parameter vector th [11]."""
    out = []
    for p, x in zip(pri, th):
        if p.kind == synth.UNIFORM:
            out.append((x - p.lo) / (p.hi - p.lo))
        elif p.kind == synth.POWERLAW:
            e = p.alpha + 1
            out.append((x ** e - p.lo ** e) / (p.hi ** e - p.lo ** e))
        elif p.kind == synth.SINE:
            out.append((math.cos(p.lo) - math.cos(x)) / (math.cos(p.lo) - math.cos(p.hi)))
        elif p.kind == synth.COSINE:
            out.append((math.sin(x) - math.sin(p.lo)) / (math.sin(p.hi) - math.sin(p.lo)))
    return np.array(out)


# ------------------------------------------------------------------ inputs
_GRID = {}


def _event(c, seed, index=0):
    """(workload, event, priors): the injection of the workload in noise of the seed."""
    w = replace(synth.workload(c["w"]), f_max=c["f_max"], seed=seed % (1 << 31), precision=c["prec"], noise=True)
    if "n_live" in c:
        w = synth.shrink(w, n_live=c["n_live"], num_delete=max(1, c["n_live"] // 2))

    def project(ev, i, th):
        key = (c["w"], c["f_max"], tuple(th))
        if key not in _GRID:
            _GRID.clear()
            geo, f, _, _ = _torch_event(ev)
            t = torch.tensor(np.asarray(th), dtype=torch.float64, device=DEV)[None]
            _GRID[key] = _strain(geo, t, f, w.waveform)[0].cpu().numpy()
        return _GRID[key][i]

    ev = synth.make_event(w, project, lambda a, b, psd, df: float(np.sum((a.conj() * b).real * 4 * df / psd)), index)
    return w, ev, synth.priors_with_injection(w, ev)


def _points(w, ev, pri, n, seed, spread):
    """n unit-cube points about the injection: `spread` of the cube wide (1: the prior)."""
    rng = np.random.default_rng([seed, 17])
    v = rng.random((n, w.n_dim))
    mid = np.clip(_unit(pri, ev.theta_inj), 0.02, 0.98)
    x = v if spread >= 1.0 else np.clip(mid * (1 - spread), 0.0, 1 - spread) + spread * v
    return torch.tensor(np.clip(x, 1e-6, 1 - 1e-6), device=DEV)


def _edges(ev, eps):
    """Coarse-bin edges by the largest phase difference of Zackay, Dai & Venumadhav 2018."""
    f = synth.frequencies(ev.f_min, ev.df, ev.n_bins)
    d = sum(2 * math.pi * math.copysign(1.0, g) * (f / (f[0] if g < 0 else f[-1])) ** g
            for g in (-5 / 3, -2 / 3, 1.0, 5 / 3, 7 / 3))
    out = [0]
    for k in range(1, ev.n_bins):
        if abs(d[k] - d[out[-1]]) > eps:
            out.append(k)
    return np.array(out + [ev.n_bins], dtype=np.int32)


def _walk_inputs(c, seed):
    w, ev, pri = _event(c, seed)
    edges = _edges(ev, c["relbin"]) if c["relbin"] else None
    ll = _Exact(ev, w.waveform, edges)
    u = _points(w, ev, pri, w.n_live, seed, c["spread"])
    lnl, order = torch.sort(ll(_theta(pri, u)))
    u, k = u[order].contiguous(), w.num_delete
    pick = torch.tensor(np.random.default_rng([seed, 18]).integers(0, w.n_live - k, k), device=DEV)
    return dict(w=w, ev=ev, pri=pri, ll=ll, edges=edges, live=u[k:].contiguous(), u0=u[k:][pick].contiguous(),
                l0=lnl[k:][pick].contiguous(), star=float(lnl[k - 1]), steps=c["steps"])


def _lnl_theta(c, seed, w, ev, pri):
    half = c["n"] // 2
    u = torch.cat([_points(w, ev, pri, c["n"] - half, seed, 1.0), _points(w, ev, pri, half, seed + 1, 0.05)])
    return _theta(pri, u).contiguous()


class _Handle:
    """A handle that is freed with its last reference."""

    def __init__(self, configs, events):
        self.h = gwns.ns_init(configs, events)

    def __del__(self):
        gwns.ns_free(self.h)


def _flow_points(c, seed):
    w, ev, pri = _event(c, seed)
    rng = np.random.default_rng([seed, 19])
    z = rng.standard_normal((c["n"], w.n_dim))
    z = 0.7 * z + 0.5 * np.roll(z, 1, 1) + 0.2 * (z ** 2 - 1)          # correlated and skewed, as a live set is
    return w, ev, pri, 1 / (1 + np.exp(-z))


def _flow_weights(c, seed, D):
    rng = np.random.default_rng([seed, 20])
    return [[rng.uniform(-1, 1, (128, D)) / math.sqrt(D), np.zeros(128), rng.uniform(-1, 1, (128, 128)) / math.sqrt(128),
             np.zeros(128), 0.02 * rng.uniform(-1, 1, (2 * D, 128)), np.zeros(2 * D)] for _ in range(c["layers"])]


def prepare(c, seed):
    kind = c["kind"]
    if kind == "run":
        evs = [_event(c, seed + 7 * i, i) for i in range(c["events"])]
        return dict(kind=kind, n=c["batches"] or 1000000, rows=0 if c["batches"] else 100 * c["n_live"],
                    configs=[gwns.make_config(w, pri) for w, _, pri in evs], events=[e for _, e, _ in evs])
    if kind == "flow":
        w, ev, pri, u = _flow_points(c, seed)
        flat = np.concatenate([a.ravel() for layer in _flow_weights(c, seed, w.n_dim) for a in layer]).astype(np.float32)
        h = _Handle([gwns.make_config(w, pri, p_flow=0.5, flow_layers=c["layers"])], [ev])
        return dict(kind=kind, h=h, u=u, flat=flat, epochs=c["epochs"], D=w.n_dim, mu=np.zeros(w.n_dim), sigma=np.ones(w.n_dim))
    if kind == "walk":
        s = _walk_inputs(c, seed)
        s["h"] = _Handle([gwns.make_config(s["w"], s["pri"])], [s["ev"]])
        if s["edges"] is not None:
            gwns.ns_relbin_set(s["h"].h, 0, s["edges"], s["ev"].theta_inj)
        n = s["u0"].shape[0]
        s["out"] = [torch.empty_like(s["u0"]), torch.empty_like(s["l0"]), torch.zeros(n, dtype=torch.int32, device=DEV),
                    torch.zeros(n, dtype=torch.int32, device=DEV)]
        return dict(s, kind=kind, ll=None)
    w, ev, pri = _event(c, seed)
    s = dict(kind=kind, h=_Handle([gwns.make_config(w, pri)], [ev]), theta=_lnl_theta(c, seed, w, ev, pri))
    if kind == "wave":
        shape = (c["n"], len(ev.detectors), ev.n_bins)
        s["out"] = [torch.empty(shape, dtype=torch.float64, device=DEV) for _ in range(2)]
    else:
        s["out"] = [torch.empty(c["n"], dtype=torch.float64, device=DEV)]
    return s


def run(s):
    kind = s["kind"]
    if kind == "lnl":
        gwns.ns_likelihood_batch(s["h"].h, 0, s["theta"], s["out"][0])
        return s["out"]
    if kind == "wave":
        gwns.ns_waveform(s["h"].h, 0, s["theta"], *s["out"])
        return s["out"]
    if kind == "walk":
        gwns.ns_walk_batch(s["h"].h, 0, s["live"], s["u0"], s["l0"], s["star"], s["steps"], 3, 0, *s["out"])
        return s["out"]
    if kind == "flow":
        h = s["h"].h
        gwns.ns_flow_set(h, 0, s["flat"], s["mu"], s["sigma"])
        losses = gwns.ns_flow_train(h, 0, s["u"], s["epochs"])
        return [losses, *gwns.ns_flow_get(h, 0, s["D"])]
    h = gwns.ns_init(s["configs"], s["events"])
    try:
        n = len(s["events"])
        _, prog = gwns.ns_step(h, s["n"], n)
        out = []
        for e in range(n):
            lz, err, info, n_like = gwns.ns_evidence(h, e)
            theta, logw = gwns.ns_posterior(h, e)
            if s["rows"]:                          # how many points a run to its stopping rule ends with varies
                theta = np.concatenate([theta, np.zeros((s["rows"] - len(theta), 11))])
                logw = np.concatenate([logw, np.zeros(s["rows"] - len(logw))])
            out.append([lz, err, info, n_like, prog[e]["iterations"], prog[e]["n_steps"], prog[e]["lnl_star"], theta, logw])
        return out
    finally:
        gwns.ns_free(h)


# ------------------------------------------------------------------ work
def _bins(c):
    """(grid bins, detectors, active bins of the injection)."""
    w = synth.workload(c["w"])
    n = synth.n_bins_for(w.f_min, c["f_max"], w.df)
    q = w.injection[1]
    m = w.injection[0] * (q / (1 + q) ** 2) ** -0.6 * MSUN_S
    cut = 1 / (6 ** 1.5 * math.pi * m) if w.waveform == synth.TAYLORF2 else X_CUT / m
    return n, len(w.detectors), max(1, min(n, int((cut - w.f_min) / w.df)))


def work(c):
    """Operations per (evaluation, active bin) as the method needs them: a basis sum of 8 to 11 terms
    for the phase, the amplitude, and per detector the time shift, one sincos, the projection and the sum."""
    n_bins, nd, active = _bins(c)
    per_bin, grid = 35.0 + 22.0 * nd, n_bins * (8.0 * 8 + nd * 24.0)
    D = synth.workload(c["w"]).n_dim
    if c["kind"] == "lnl":
        return {"bytes": grid + c["n"] * 96.0, "flops": c["n"] * active * per_bin}
    if c["kind"] == "wave":
        return {"bytes": grid + c["n"] * (88.0 + 16.0 * nd * n_bins), "flops": c["n"] * active * per_bin}
    if c["kind"] == "flow":
        layer = 2.0 * (D * 128 + 128 * 128 + 2 * D * 128)
        return {"bytes": 8.0 * c["n"] * D + 3 * 4 * 20000.0 * c["layers"], "flops": 3.0 * layer * c["layers"] * c["n"] * c["epochs"]}
    # about one step in four of a walk stays in the cube and is evaluated
    if c["kind"] == "walk":
        k = max(1, c["n_live"] // 2)
        bins = 130.0 if c["relbin"] else active
        return {"bytes": grid + 16.0 * (c["n_live"] - k + 2 * k) * D, "flops": 0.25 * k * c["steps"] * bins * per_bin}
    batches, steps = (c["batches"] or 30), 240.0 if D > 4 else 80.0
    evals = c["n_live"] + 0.25 * batches * steps * (c["n_live"] // 2)
    return {"bytes": c["events"] * (grid + 8.0 * D * c["n_live"] * (1 + batches)), "flops": c["events"] * evals * active * per_bin}


# ------------------------------------------------------------------ 64-bit outputs
_M32 = np.uint64(0xFFFFFFFF)


def _mulhi(a, b):
    al, ah, bl, bh = a & _M32, a >> np.uint64(32), np.uint64(b & 0xFFFFFFFF), np.uint64(b >> 32)
    mid = (al * bl >> np.uint64(32)) + (al * bh & _M32) + (ah * bl & _M32)
    return ah * bh + (al * bh >> np.uint64(32)) + (ah * bl >> np.uint64(32)) + (mid >> np.uint64(32))


def _philox(c0, c1, c2, c3, k0, k1):
    """Philox4x64-10 (Salmon et al. 2011) on arrays of counters."""
    m0, m1 = 0xD2E7470EE14C6C93, 0xCA5A826395121157
    c = [np.broadcast_to(np.asarray(x, dtype=np.uint64), np.broadcast(c0, c1).shape) for x in (c0, c1, c2, c3)]
    for _ in range(10):
        h0, l0, h1, l1 = _mulhi(c[0], m0), c[0] * np.uint64(m0), _mulhi(c[2], m1), c[2] * np.uint64(m1)
        c = [h1 ^ c[1] ^ np.uint64(k0), l1, h0 ^ c[3] ^ np.uint64(k1), l0]
        k0, k1 = (k0 + 0x9E3779B97F4A7C15) & (2 ** 64 - 1), (k1 + 0xBB67AE8584CAA73B) & (2 ** 64 - 1)
    return c


def _open(x):
    return ((x >> np.uint64(12)).astype(np.float64) + 0.5) / 4503599627370496.0


def _walk_exact(s, seed):
    n, D = s["u0"].shape
    n_s, T = s["live"].shape[0], s["steps"]
    t, j = np.meshgrid(np.arange(T, dtype=np.uint64), np.arange(n, dtype=np.uint64), indexing="ij")
    A = _philox(t, j, 3, 0, s["w"].seed, 0)
    B = _philox(t, j, 3, 1, s["w"].seed, 0)
    a, b = _mulhi(A[0], n_s).astype(np.int64), _mulhi(A[1], n_s - 1).astype(np.int64)
    b = b + (b >= a)
    g = -0.25 * np.log(_open(B[0]) * _open(B[1]) * _open(B[2]) * _open(B[3]))
    sc = np.where(A[2] >> np.uint64(63) == 1, 1.0, 2.38 / math.sqrt(2 * D) * g)
    a, b, sc = (torch.tensor(x, device=DEV) for x in (a, b, sc))
    per = torch.tensor([p.periodic for p in s["pri"] if p.kind != synth.FIXED], device=DEV)
    u, lnl = s["u0"].clone(), s["l0"].clone()
    for t in range(T):
        p = u + sc[t][:, None] * (s["live"][a[t]] - s["live"][b[t]])
        p = torch.where(per, p - torch.floor(p), p)
        rows = ((p >= 0) & (p <= 1)).all(1).nonzero()[:, 0]
        if rows.numel():
            v = s["ll"](_theta(s["pri"], p[rows]))
            up = v > s["star"]
            u[rows[up]], lnl[rows[up]] = p[rows[up]], v[up]
    return [u, lnl, None, None]


def _flow_exact(c, seed):
    """Maximum-likelihood training in 64 bits (the library's matrix products take 16-bit operands)."""
    w, _, _, u = _flow_points(c, seed)
    D, L = w.n_dim, c["layers"]
    par = [torch.tensor(np.asarray(a, dtype=np.float32).astype(np.float64), device=DEV, requires_grad=True)
           for layer in _flow_weights(c, seed, D) for a in layer]
    u = torch.tensor(u, device=DEV)
    lg = torch.log(u) - torch.log1p(-u)
    mu, sg = lg.mean(0), lg.std(0, unbiased=False)
    base = -(torch.log(u) + torch.log1p(-u)).sum(1) - torch.log(sg).sum()
    m1, m2 = [torch.zeros_like(p) for p in par], [torch.zeros_like(p) for p in par]
    losses = []
    for step in range(1, c["epochs"] + 1):
        z, ld = (lg - mu) / sg, base
        for l in range(L):
            W1, b1, W2, b2, W3, b3 = par[6 * l:6 * l + 6]
            m = ((torch.arange(D, device=DEV) + l) % 2 == 0).double()
            o = torch.tanh(torch.tanh((m * z) @ W1.T + b1) @ W2.T + b2) @ W3.T + b3
            s, t = (1 - m) * 2 * torch.tanh(o[:, :D] / 2), (1 - m) * o[:, D:]
            z, ld = m * z + (1 - m) * (z * torch.exp(s) + t), ld + s.sum(1)
        loss = -(ld - 0.5 * (z * z).sum(1) - 0.5 * D * math.log(2 * math.pi)).mean()
        losses.append(float(loss))
        with torch.no_grad():
            for p, g, a, b in zip(par, torch.autograd.grad(loss, par), m1, m2):
                a.mul_(0.9).add_(0.1 * g)
                b.mul_(0.999).add_(0.001 * g * g)
                p -= 3e-3 * (a / (1 - 0.9 ** step)) / (torch.sqrt(b / (1 - 0.999 ** step)) + 1e-8)
    flat = torch.cat([p.detach().ravel() for p in par])
    return [np.array(losses), flat, mu, sg]


def exact(c, seed):
    if c["kind"] == "run":
        return None                                # a whole run: minutes in plain 64 bits
    if c["kind"] == "flow":
        return _flow_exact(c, seed)
    if c["kind"] == "walk":
        s = _walk_inputs(c, seed)
        evals = 0.3 * s["u0"].shape[0] * c["steps"]
        if evals * _bins(c)[0] > 1e10:
            return None                            # over 20 s in plain 64 bits
        return _walk_exact(s, seed)
    w, ev, pri = _event(c, seed)
    th = _lnl_theta(c, seed, w, ev, pri)
    if c["kind"] == "lnl":
        return [_Exact(ev, w.waveform)(th)]
    geo, f, _, _ = _torch_event(ev)
    h = torch.cat([_strain(geo, t, f, w.waveform) for t in th.split(4)])
    return [h.real.contiguous(), h.imag.contiguous()]
