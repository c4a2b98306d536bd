"""Workloads that stand for the library's use, each through its public entry points.

A case is a dict of plain values: the entry point (``call``), the event (one of the five
synthetic workloads' recipes: source class, detectors, duration, band), the batch, the
precision and the launch shape that the program has chosen.  ``prepare`` makes the event,
its context and the batch from the seed; ``run`` is one call; ``exact`` is the same
likelihood and gradient written out per bin in plain FP64 torch.
"""
import math

import numpy as np
import torch

from paper_1909_11873_gb300 import gwl
from paper_1909_11873_gb300 import inputs as I

SOLAR_TIME = 4.925490947e-6      # G M_sun / c^3 [s]
LIGHT = 299792458.0              # [m/s]
MPC = 3.085677581491367e22       # [m]


def listed():
    return [
        # an external sampler on the host hands over a few points at a time in pinned buffers: the smallest call
        dict(name="host_4s_16", call="host", source="c1", n_det=1, T=4.0, f_high=512.0, B=16, prec="mixed",
             layout="auto", window=0),
        # one parallel round's proposals of the 1-detector 4 s event, two-window cuts among them
        dict(name="lnl_4s_1024", call="loglike", source="c1", n_det=1, T=4.0, f_high=512.0, B=1024, prec="mixed",
             layout="auto", window=0),
        # the benchmark's batch: 3 detectors, 8 s BBH, the shape that the autotuner settles on
        dict(name="lnl_8s_8192", call="loglike", source="bbh", n_det=3, T=8.0, f_high=1024.0, B=8192, prec="mixed",
             layout="warp", window=704),
        # long neutron-star signals: 260 thousand bins per detector, one proposal per lane
        dict(name="lnl_128s_2048", call="loglike", source="bns", n_det=3, T=128.0, f_high=2048.0, B=2048,
             prec="mixed", layout="lane", window=1280),
        # the FP64 mode, as used to check a posterior
        dict(name="lnl_fp64_8s_1021", call="loglike", source="bbh", n_det=3, T=8.0, f_high=1024.0, B=1021,
             prec="fp64", layout="auto", window=0),
        # with the calibration model, 71 parameters per row
        dict(name="cal_8s_4096", call="loglike", source="bbh", n_det=3, T=8.0, f_high=1024.0, B=4096, prec="mixed",
             layout="warp", window=704, nodes=10),
        # likelihood and gradient of one batch
        dict(name="grad_8s_4096", call="grad", source="bbh", n_det=3, T=8.0, f_high=1024.0, B=4096, prec="mixed",
             layout="auto", window=0),
        # gradient with the calibration model: 71 derivatives per row
        dict(name="calgrad_8s_2048", call="grad", source="bbh", n_det=3, T=8.0, f_high=1024.0, B=2048, prec="mixed",
             layout="auto", window=0, nodes=10),
        # a round's constrained random walks (Algorithm 1's parallel step) driven from the caller's own sampler
        dict(name="walk_4s_250x20", call="replace", source="c1", n_det=1, T=4.0, f_high=512.0, K=250, n=250,
             walk=20, prec="mixed", kind="random"),
        # the gradient-informed walk in 11 dimensions
        dict(name="galilean_8s_250x10", call="replace", source="bbh", n_det=3, T=8.0, f_high=1024.0, K=500, n=250,
             walk=10, prec="mixed", kind="galilean"),
        # a whole nested-sampling run on the device
        dict(name="ns_run_4s_250", call="ns_run", source="c1", n_det=1, T=4.0, f_high=512.0, K=250, n=250, walk=20,
             prec="mixed"),
        # a batch of events of uneven durations
        dict(name="multi_12x500", call="multi", n_events=12, n_det=3, f_high=1024.0, n_per=500, prec="mixed"),
    ]


def _logint(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """One more case of the same ranges."""
    call = rng.choice(["host", "loglike", "loglike", "loglike", "loglike", "cal", "grad", "grad", "calgrad", "replace",
                       "galilean", "ns_run", "multi"])
    if call == "ns_run":
        K = rng.randint(100, 250)
        return dict(call="ns_run", source="c1", n_det=1, T=4.0, f_high=512.0, K=K, n=rng.randint(K, 2 * K),
                    walk=rng.randint(10, 20), prec="mixed")
    if call == "multi":
        return dict(call="multi", n_events=rng.randint(2, 12), n_det=rng.choice([2, 3]), f_high=1024.0,
                    n_per=_logint(rng, 50, 500), prec="mixed")
    if call in ("replace", "galilean"):
        src = "c1" if call == "replace" and rng.random() < 0.5 else "bbh"
        base = dict(source="c1", n_det=1, T=4.0, f_high=512.0) if src == "c1" else \
            dict(source="bbh", n_det=rng.choice([2, 3]), T=rng.choice([4.0, 8.0]), f_high=1024.0)
        n = _logint(rng, 25, 250 if call == "galilean" else 1000)
        return dict(base, call="replace", K=rng.randint(200, 500), n=n,
                    walk=rng.randint(5, 10 if call == "galilean" else 25), prec="mixed",
                    kind="galilean" if call == "galilean" else "random")
    if call in ("cal", "calgrad"):
        return dict(call="grad" if call == "calgrad" else "loglike", source="bbh", n_det=rng.choice([1, 2, 3, 4]),
                    T=rng.choice([4.0, 8.0]), f_high=1024.0,
                    B=_logint(rng, 64, 2048 if call == "calgrad" else 4096), prec="mixed", layout="auto", window=0,
                    nodes=rng.randint(5, 10))
    if call == "host":
        src = rng.choice(["c1", "bbh"])
        base = dict(source="c1", n_det=1, T=4.0, f_high=512.0) if src == "c1" else \
            dict(source="bbh", n_det=rng.choice([2, 3]), T=8.0, f_high=1024.0)
        return dict(base, call="host", B=_logint(rng, 1, 1024), prec="mixed", layout="auto", window=0)
    if call == "grad":
        return dict(call="grad", source="bbh", n_det=rng.choice([1, 2, 3, 4]), T=rng.choice([4.0, 8.0, 16.0]),
                    f_high=1024.0, B=_logint(rng, 16, 4096), prec="mixed", layout="auto", window=0)
    what = rng.choice(["c1", "bbh", "bbh", "bns", "fp64"])
    if what == "c1":
        return dict(call="loglike", source="c1", n_det=1, T=4.0, f_high=512.0, B=_logint(rng, 1, 4096), prec="mixed",
                    layout="auto", window=0)
    if what == "bbh":
        layout = rng.choice(["auto", "warp"])
        return dict(call="loglike", source="bbh", n_det=rng.choice([1, 2, 3, 4]), T=rng.choice([4.0, 8.0, 16.0]),
                    f_high=1024.0, B=_logint(rng, 32, 8192), prec="mixed", layout=layout,
                    window=32 * rng.randint(20, 26) if layout == "warp" else 0)
    if what == "bns":
        T = rng.choice([32.0, 64.0, 128.0])
        return dict(call="loglike", source="bns", n_det=rng.choice([2, 3]), T=T, f_high=rng.choice([1024.0, 2048.0]),
                    B=_logint(rng, 64, 2048), prec="mixed", layout=rng.choice(["auto", "lane"]), window=1280)
    return dict(call="loglike", source="bbh", n_det=rng.choice([1, 2, 3]), T=rng.choice([4.0, 8.0]), f_high=1024.0,
                B=_logint(rng, 32, 1024), prec="fp64", layout="auto", window=0)


# ---------------------------------------------------------------- the model in plain FP64 torch
def _phase_terms(th, f):
    """[n, M] phase at each detector-independent frequency [rad] and [n, M] in-band mask, for rows th [n, 11]."""
    mc, q, c1, c2 = (th[:, k:k + 1] for k in range(4))
    eta = q / (1.0 + q) ** 2
    delta = (1.0 - q) / (1.0 + q)
    m1, m2 = 1.0 / (1.0 + q), q / (1.0 + q)
    cs, ca = 0.5 * (c1 + c2), 0.5 * (c1 - c2)
    a = math.pi * mc * eta ** -0.6 * SOLAR_TIME  # pi M
    v = (a * f) ** (1.0 / 3.0)
    lv = torch.log(a * f) / 3.0
    beta = (113.0 / 12.0 * m1 ** 2 + 25.0 / 4.0 * eta) * c1 + (113.0 / 12.0 * m2 ** 2 + 25.0 / 4.0 * eta) * c2
    sigma = 79.0 / 8.0 * eta * c1 * c2
    gam = (732985.0 / 2268.0 - 24260.0 / 81.0 * eta - 340.0 / 9.0 * eta ** 2) * cs + \
        (732985.0 / 2268.0 + 140.0 / 9.0 * eta) * delta * ca
    p2 = 20.0 / 9.0 * (743.0 / 336.0 + 11.0 / 4.0 * eta)
    p3 = 4.0 * beta - 16.0 * math.pi
    p4 = 10.0 * (3058673.0 / 1016064.0 + 5429.0 / 1008.0 * eta + 617.0 / 144.0 * eta ** 2) - 10.0 * sigma
    p5 = (math.pi * (38645.0 / 756.0 - 65.0 / 9.0 * eta) - gam) * (1.0 + 3.0 * lv + 1.5 * math.log(6.0))
    p6 = 11583231236531.0 / 4694215680.0 - 640.0 / 3.0 * math.pi ** 2 - 6848.0 / 21.0 * 0.5772156649015329 + \
        eta * (-15737765635.0 / 3048192.0 + 2255.0 / 12.0 * math.pi ** 2) + 76055.0 / 1728.0 * eta ** 2 - \
        127825.0 / 1296.0 * eta ** 3 + math.pi * (2270.0 / 3.0 * delta * ca + (2270.0 / 3.0 - 520.0 * eta) * cs) - \
        6848.0 / 21.0 * (math.log(4.0) + lv)
    p7 = math.pi * (77096675.0 / 254016.0 + 378515.0 / 1512.0 * eta - 74045.0 / 756.0 * eta ** 2) + \
        (-25150083775.0 / 3048192.0 + 10566655595.0 / 762048.0 * eta - 1042165.0 / 3024.0 * eta ** 2 +
         5345.0 / 36.0 * eta ** 3) * cs + \
        delta * (-25150083775.0 / 3048192.0 + 26804935.0 / 6048.0 * eta - 1985.0 / 48.0 * eta ** 2) * ca
    s = 1.0 + v ** 2 * (p2 + v * (p3 + v * (p4 + v * (p5 + v * (p6 + v * p7)))))
    band = f <= 1.0 / (6.0 ** 1.5 * a.detach())
    return 3.0 / (128.0 * eta * v ** 5) * s, band


def _detector(th, g, gmst):
    """Antenna response (plus, cross amplitudes) and the arrival delay of one detector: [n] each."""
    inc, psi, ra, dec = th[:, 5], th[:, 6], th[:, 7], th[:, 8]
    lam = ra - gmst
    sl, cl, sd, cd, sp, cp = (fn(x) for x in (lam, dec, psi) for fn in (torch.sin, torch.cos))
    east = (-sl, cl, torch.zeros_like(sl))
    north = (-sd * cl, -sd * sl, cd)
    X = [cp * e + sp * n for e, n in zip(east, north)]
    Y = [-sp * e + cp * n for e, n in zip(east, north)]
    dot = lambda u, w: sum(float(a) * b for a, b in zip(u, w))  # noqa: E731
    xX, xY, yX, yY = dot(g[3:6], X), dot(g[3:6], Y), dot(g[6:9], X), dot(g[6:9], Y)
    fp = 0.5 * ((xX ** 2 - xY ** 2) - (yX ** 2 - yY ** 2))
    fx = xX * xY - yX * yY
    ci = torch.cos(inc)
    delay = -dot(g[0:3], (cd * cl, cd * sl, sd)) / LIGHT
    return fp * 0.5 * (1.0 + ci ** 2), -fx * ci, delay


def _template(ev, th, cal=None, m_max=None):
    """Real and imaginary template per detector [n, M] of rows th [n, 11] (a generator over detectors)."""
    f = torch.as_tensor(ev.freqs[:m_max], device=th.device)[None, :]
    pn, band = _phase_terms(th, f)
    amp = math.sqrt(5.0 / 24.0) * math.pi ** (-2.0 / 3.0) * (th[:, 0] * SOLAR_TIME) ** (5.0 / 6.0) * LIGHT / \
        (th[:, 4] * MPC)
    af = torch.where(band, amp[:, None] * f ** (-7.0 / 6.0), torch.zeros((), dtype=f.dtype, device=f.device))
    for d in range(ev.geom.shape[0]):
        pr, pi, dt = _detector(th, ev.geom[d], ev.gmst)
        psi = 2.0 * math.pi * f * (ev.t_ref + th[:, 9] + dt)[:, None] - (th[:, 10] + 0.25 * math.pi)[:, None] + pn
        a = af
        if cal is not None:
            a = af * (1.0 + cal[d][0])
            psi = psi - cal[d][1]
        c, s = torch.cos(psi), torch.sin(psi)
        yield a * (pr[:, None] * c + pi[:, None] * s), a * (pi[:, None] * c - pr[:, None] * s)


def _spline_basis(nodes, freqs):
    """[n_nodes, M] cardinal functions of the natural cubic spline in ln f."""
    x, t = np.log(np.asarray(nodes)), np.log(np.asarray(freqs))
    n = x.size
    h = np.diff(x)
    A, R = np.eye(n), np.zeros((n, n))
    for k in range(1, n - 1):
        A[k, k - 1:k + 2] = h[k - 1], 2.0 * (h[k - 1] + h[k]), h[k]
        R[k, k - 1:k + 2] = 6.0 / h[k - 1], -6.0 / h[k - 1] - 6.0 / h[k], 6.0 / h[k]
    m = np.linalg.solve(A, R)  # curvatures at the nodes of each cardinal function
    i = np.clip(np.searchsorted(x, t, side="right") - 1, 0, n - 2)
    u = (t - x[i]) / h[i]
    y = np.eye(n)
    w = h[i] ** 2 / 6.0
    return ((1 - u)[:, None] * y[i] + u[:, None] * y[i + 1] + (w * ((1 - u) ** 3 - (1 - u)))[:, None] * m[i] +
            (w * (u ** 3 - u))[:, None] * m[i + 1]).T


def _lnl(ev, rows, basis=None):
    """lnL [n] of rows [n, D (+ calibration)] on one event."""
    smp = ev.sampling
    D = smp.D
    pos = {int(p): i for i, p in enumerate(smp.param_map)}
    th = torch.stack([rows[:, pos[k]] if k in pos else torch.full_like(rows[:, 0], float(smp.fixed[k]))
                      for k in range(11)], dim=1)
    with torch.no_grad():
        eta = th[:, 1] / (1.0 + th[:, 1]) ** 2
        top = float((1.0 / (6.0 ** 1.5 * math.pi * th[:, 0] * eta ** -0.6 * SOLAR_TIME)).max())
    m_max = max(1, min(ev.M, int((top - ev.freqs[0]) * ev.T) + 2))
    cal = None
    if basis is not None:
        nn = basis.shape[0]
        y = rows[:, D:].reshape(rows.shape[0], ev.n_det, 2, nn)
        cal = [(y[:, d, 0] @ basis[:, :m_max], y[:, d, 1] @ basis[:, :m_max]) for d in range(ev.n_det)]
    out = torch.zeros_like(rows[:, 0])
    for d, (hr, hi) in enumerate(_template(ev, th, cal, m_max)):
        w = torch.as_tensor(4.0 * ev.df / ev.psd[d, :m_max], device=rows.device)
        dr = torch.as_tensor(np.ascontiguousarray(ev.strain[d, :m_max].real), device=rows.device)
        di = torch.as_tensor(np.ascontiguousarray(ev.strain[d, :m_max].imag), device=rows.device)
        out = out + ((hr * (dr - 0.5 * hr) + hi * (di - 0.5 * hi)) * w).sum(dim=1)
    return out


def _lnl_chunks(ev, rows, basis=None, gradient=False):
    step = max(1, min(rows.shape[0], int(2e7 / ev.M)))
    ls, gs = [], []
    for k in range(0, rows.shape[0], step):
        x = rows[k:k + step].clone().requires_grad_(gradient)
        with torch.set_grad_enabled(gradient):
            v = _lnl(ev, x, basis)
            if gradient:
                gs.append(torch.autograd.grad(v.sum(), x)[0])
        ls.append(v.detach())
    return (torch.cat(ls), torch.cat(gs)) if gradient else torch.cat(ls)


# ---------------------------------------------------------------- events and batches
def _waveform(ev, th):
    x = torch.as_tensor(np.asarray(th)[None], device="cuda")
    return np.stack([(hr[0] + 1j * hi[0]).cpu().numpy() for hr, hi in _template(ev, x)])


def _snr2(ev, th):
    x = torch.as_tensor(np.asarray(th)[None], device="cuda")
    s = 0.0
    for d, (hr, hi) in enumerate(_template(ev, x)):
        s += float(((hr ** 2 + hi ** 2) * torch.as_tensor(4.0 * ev.df / ev.psd[d], device="cuda")).sum())
    return s


def _event(source, n_det, T, f_high, seed):
    cfg = dict(n_det=n_det, T=T, f_low=20.0, f_high=f_high, noise=source != "c1", source=source,
               gmst=0.3 if source == "c1" else 1.7)
    return I.make_event(source, seed, _waveform, _snr2, cfg=cfg)


def _case_event(case, seed):
    return _event(case["source"], case["n_det"], case["T"], case["f_high"], seed)


def _rows(case, ev, seed):
    """[B, D (+ calibration)] proposals: half prior draws, half near the injection (all prior draws on the 4 s event)."""
    th = I.proposals(ev, case["B"], seed + 1, local_fraction=0.0 if case["source"] == "c1" else 0.5)
    rows = I.reduced(th, ev.sampling)
    if case.get("nodes"):
        cal = I.draw_calibration(np.random.default_rng(seed + 7), case["B"], ev.n_det, case["nodes"])
        rows = np.ascontiguousarray(np.concatenate([rows, cal], axis=1))
    return rows


def _nodes(case, ev):
    return I.cal_node_freqs(float(ev.freqs[0]), float(ev.freqs[-1]), case["nodes"]) if case.get("nodes") else None


def _multi_events(case, seed):
    """Events of 4 to 128 s, black holes and neutron stars, their durations spread over the whole range."""
    rng = np.random.default_rng(seed)
    out = []
    for e in range(case["n_events"]):
        T = I.C4_DURATIONS[e % len(I.C4_DURATIONS)]
        src = "bbh" if rng.uniform() < 0.5 else "bns"
        ev = _event(src, case["n_det"], T, case["f_high"], int(rng.integers(1 << 31)))
        out.append((ev, I.reduced(I.proposals(ev, case["n_per"], int(rng.integers(1 << 30))), ev.sampling)))
    return out


def _prec(case):
    return gwl.GWL_FP64 if case["prec"] == "fp64" else gwl.GWL_MIXED


def _context(case, ev):
    ctx = gwl.Context.from_event(ev, _prec(case))
    if case.get("nodes"):
        ctx.gwl_set_calibration(_nodes(case, ev))
    if case.get("layout") == "warp":
        ctx.gwl_set_tuning(window=case["window"], ctas_per_sm=2, bin_kernel=gwl.GWL_BINS_WARP)
    elif case.get("layout") == "lane":
        ctx.gwl_set_tuning(window=case["window"], ctas_per_sm=2, bin_kernel=gwl.GWL_BINS_LANE)
    return ctx


def _prior_points(smp, n, rng):
    u = rng.uniform(0.0, 1.0, (n, smp.D))
    th = np.empty_like(u)
    for i in range(smp.D):
        lo, hi, k = smp.lo[i], smp.hi[i], smp.kind[i]
        if k == I.VOLUME:
            th[:, i] = np.cbrt(lo ** 3 + u[:, i] * (hi ** 3 - lo ** 3))
        elif k == I.SINE:
            th[:, i] = np.arccos(1.0 - 2.0 * u[:, i])
        elif k == I.COSINE:
            th[:, i] = np.arcsin(2.0 * u[:, i] - 1.0)
        else:
            th[:, i] = lo + u[:, i] * (hi - lo)
    return u, th


def prepare(case, seed):
    call = case["call"]
    if call == "multi":
        evs = _multi_events(case, seed)
        ctxs = [_context(case, ev) for ev, _ in evs]
        theta = torch.from_numpy(np.concatenate([r for _, r in evs])).cuda()
        return dict(call=call, multi=gwl.MultiContext(ctxs), theta=theta,
                    out=torch.empty(theta.shape[0], dtype=torch.float64, device="cuda"))
    ev = _case_event(case, seed)
    ctx = _context(case, ev)
    if call in ("loglike", "grad"):
        return dict(call=call, ctx=ctx, theta=torch.from_numpy(_rows(case, ev, seed)).cuda())
    if call == "host":
        theta = torch.from_numpy(_rows(case, ev, seed)).pin_memory()
        out = torch.empty(case["B"], dtype=torch.float64).pin_memory()
        return dict(call=call, ctx=ctx, theta=theta.numpy(), out=out.numpy(), keep=(theta, out))
    if call == "ns_run":
        return dict(call=call, ctx=ctx, K=case["K"], n=case["n"], walk=case["walk"], seed=seed + 17)
    # a live set in mid-run: the best K of 4 K prior points, their covariance's Cholesky factor
    if case["kind"] == "galilean":
        ctx.gwl_set_walk(gwl.GWL_WALK_GALILEAN)
    K, n, D = case["K"], case["n"], ev.sampling.D
    u, th = _prior_points(ev.sampling, 4 * K, np.random.default_rng(seed + 3))
    l = gwl.loglike(ctx, torch.from_numpy(th).cuda())
    best = torch.sort(torch.topk(l, K).indices).values
    live_u = torch.from_numpy(u).cuda()[best].contiguous()
    live_l = l[best].contiguous()
    chol = torch.linalg.cholesky(torch.cov(live_u.T)).contiguous()
    worst = int(torch.argmin(live_l))
    return dict(call=call, ctx=ctx, live_u=live_u, live_l=live_l, chol=chol, worst=worst, star=float(live_l[worst]),
                n=n, walk=case["walk"], seed=seed + 29,
                out_u=torch.empty((n, D), dtype=torch.float64, device="cuda"),
                out_l=torch.empty(n, dtype=torch.float64, device="cuda"),
                out_n=torch.empty(n, dtype=torch.int32, device="cuda"),
                out_s=torch.empty(n, dtype=torch.int32, device="cuda"))


def run(s):
    call = s["call"]
    if call == "loglike":
        return gwl.loglike(s["ctx"], s["theta"])
    if call == "grad":
        return gwl.grad(s["ctx"], s["theta"])
    if call == "host":
        s["ctx"].gwl_loglike_host(s["theta"], s["out"])
        return s["out"]
    if call == "multi":
        s["multi"].gwl_multi_loglike(s["theta"], s["out"])
        return s["out"]
    if call == "replace":
        s["ctx"].ns_replace(s["live_u"], s["live_l"], s["worst"], s["star"], s["seed"], 0, s["n"], s["walk"], 0.3,
                            s["chol"], s["out_u"], s["out_l"], s["out_n"], s["out_s"])
        return s["out_u"], s["out_l"], s["out_n"], s["out_s"]
    cap = 40 * s["K"]
    r = s["ctx"].ns_run(s["K"], s["n"], s["walk"], s["seed"], max_dead=cap)
    out = {k: r[k] for k in ("lnZ", "lnZ_err", "H", "n_dead", "n_proposals", "rounds", "scale", "acceptance",
                             "consumed_per_round", "dlogz")}
    for k in ("dead_lnl", "dead_logwt", "dead_u"):  # arrays of the capacity asked for, zero past the last dead point
        out[k] = np.zeros((cap,) + r[k].shape[1:])
        out[k][:r["n_dead_returned"]] = r[k]
    return out


def exact(case, seed):
    """lnL (and gradient) in FP64; the walks' and the sampler's results have no closed value."""
    call = case["call"]
    if call == "multi":
        return torch.cat([_lnl_chunks(ev, torch.from_numpy(r).cuda()) for ev, r in _multi_events(case, seed)])
    if call in ("replace", "ns_run"):
        return None
    ev = _case_event(case, seed)
    basis = torch.from_numpy(_spline_basis(_nodes(case, ev), ev.freqs)).cuda() if case.get("nodes") else None
    rows = torch.from_numpy(_rows(case, ev, seed)).cuda()
    v = _lnl_chunks(ev, rows, basis, gradient=call == "grad")
    return v.cpu().numpy() if call == "host" else v


def _mean_cut(source, T, f_high):
    """Mean in-band bins of prior draws (the cut from the total mass)."""
    rng = np.random.default_rng(5)
    mc, q = {"c1": ((8.0, 12.0), (0.5, 1.0)), "bbh": (I.BBH["mc"], I.BBH["q"]),
             "bns": (I.BNS["mc"], I.BNS["q"])}[source]
    m, r = rng.uniform(*mc, 4096), rng.uniform(*q, 4096)
    fc = 1.0 / (6.0 ** 1.5 * math.pi * m * (r / (1 + r) ** 2) ** -0.6 * SOLAR_TIME)
    return float(np.mean(np.clip(np.floor((np.minimum(fc, f_high) - 20.0) * T) + 1, 0, None)))


def work(case):
    """Bytes: parameters in, results out and the in-band data once.  Flops: the arithmetic per in-band
    (proposal, bin): the eight-term phase, and per detector the delay, sine and cosine and the complex
    multiply-add (plus the gradient's weighted sums, the calibration's splines)."""
    nd = case["n_det"]
    if case["call"] == "multi":
        cuts = [0.5 * (_mean_cut("bbh", T, case["f_high"]) + _mean_cut("bns", T, case["f_high"]))
                for T in (I.C4_DURATIONS[e % len(I.C4_DURATIONS)] for e in range(case["n_events"]))]
        return {"bytes": 96.0 * case["n_events"] * case["n_per"] + sum(cuts) * nd * 24.0,
                "flops": sum(cuts) * case["n_per"] * (17.0 + 14.0 * nd)}
    cut = _mean_cut(case["source"], case["T"], case["f_high"])
    D = 4 if case["source"] == "c1" else 11
    dim = D + 2 * case.get("nodes", 0) * nd
    per = 17.0 + 14.0 * nd
    if case.get("nodes"):
        per += 9.0 + 22.0 * nd
    if case["call"] == "grad":
        per += 16.0 + 11.0 * nd
        if case.get("nodes"):
            per += 50.0 * nd
    if case["call"] == "replace":
        rows = case["n"] * case["walk"]
        if case["kind"] == "galilean":
            per += 16.0 + 11.0 * nd
        return {"bytes": 8.0 * (dim + 1) * (case["n"] + case["K"]) + cut * nd * 24.0, "flops": rows * cut * per}
    if case["call"] == "ns_run":
        rounds = 20.0 / math.log(1.0 + case["n"] / case["K"])
        return {"bytes": 8.0 * (dim + 2) * 22.0 * case["K"] + cut * nd * 24.0,
                "flops": rounds * case["n"] * case["walk"] * cut * per}
    out = (dim + 1) if case["call"] == "grad" else 1
    return {"bytes": 8.0 * case["B"] * (dim + out) + cut * nd * 24.0, "flops": case["B"] * cut * per}
