"""The calls whose time counts: what a user of this package has the GPU do.

Every case runs through the public entry points of paper_2601_02336_gb300.api. Workloads are the ones of
paper_2601_02336_gb300.inputs (the 4-D toy signal, the 11-D binary-black-hole signal on 4 to 32 s segments, the low-mass
signal on 128 s); events, noise and parameter sets are made from the seed. Inputs (strain, ln L and gradients handed to
the sampler's calls) come from a plain torch evaluation in 64 bits below, so they do not depend on the code under test.
"""
import math

import numpy as np
import torch

from paper_2601_02336_gb300 import api, inputs

DEV = "cuda:0"
TSUN = 4.925491025543576e-6
MPC_S = 3.085677581491367e22 / 299792458.0
EARTH_S = 6.371e6 / 299792458.0

# ------------------------------------------------------------------ the cases


def listed():
    return [
        # the smallest call: ln L and gradient of the toy signal's ensemble, one launch
        dict(name="lnl_toy_128", kind="lnl", signal="toy", seconds=4, fmax=128, n=128, where="prior", precision="mixed",
             how="grad"),
        # the ordinary call: the first evaluation of an 11-D run, prior draws
        dict(name="lnl_bbh_prior_2048", kind="lnl", signal="bbh", seconds=8, fmax=1024, n=2048, where="prior",
             precision="mixed", how="grad"),
        # torch code that differentiates through ln L (forward sweep, then the adjoint); an odd count of posterior draws
        dict(name="lnl_autograd_5001", kind="lnl", signal="bbh", seconds=16, fmax=2048, n=5001, where="ball",
             precision="split", how="autograd"),
        # the largest call: 128 s of a low-mass signal, a full ensemble near the injection
        dict(name="lnl_bns_8192", kind="lnl", signal="bns", seconds=128, fmax=2048, n=8192, where="ball",
             precision="mixed", how="grad"),
        # the FP64 option: the check of a mixed result, on a part of the ensemble
        dict(name="lnl_bbh_fp64_1000", kind="lnl", signal="bbh", seconds=8, fmax=1024, n=1000, where="ball",
             precision="fp64", how="grad"),
        # the mutation of an 11-D run's first stage: near the prior, most trees reach the depth limit
        dict(name="nuts_first_2048", kind="nuts", signal="bbh", seconds=8, fmax=1024, n=2048, where="prior",
             beta=1e-4, metric="identity", depth=6, precision="mixed"),
        # a last stage with the per-particle metric, which the call before the mutation forms
        dict(name="nuts_local_2048", kind="nuts", signal="bbh", seconds=8, fmax=1024, n=2048, where="ball",
             beta=1.0, metric="local", depth=6, precision="split"),
        # the large ensemble: 16 s to 2048 Hz, covariance metric, deeper trees
        dict(name="nuts_long_16384", kind="nuts", signal="bbh", seconds=16, fmax=2048, n=16384, where="ball",
             beta=1.0, metric="covariance", depth=8, precision="mixed"),
        # the same mutation in FP64 (the reference runs a mixed evidence is checked against), odd count
        dict(name="nuts_fp64_1001", kind="nuts", signal="bbh", seconds=8, fmax=1024, n=1001, where="ball",
             beta=1.0, metric="identity", depth=6, precision="fp64"),
        # everything between two mutations: tempering root, weights, evidence, resampling, gather, local metrics
        dict(name="stage_16384", kind="stage", signal="bbh", seconds=8, fmax=1024, n=16384, beta=0.0, metric="local"),
        # one whole analysis: an SMC run and the recycling of its stages' particles
        dict(name="run_bbh_2048", kind="run", signal="bbh", seconds=8, fmax=1024, n=2048, metric="identity", depth=6,
             precision="mixed"),
        # a catalogue: eight events of 4 to 32 s and uneven particle counts in one batched run
        dict(name="batch_8_events", kind="batch", events=8, depth=8, precision="mixed"),
    ]


def _loguniform(rng, a, b):
    return int(round(math.exp(rng.uniform(math.log(a), math.log(b)))))


def draw(rng):
    """A likelihood call, a mutation or a stage of other sizes: any segment length, count, type and metric in use."""
    most = max(work(c)["flops"] for c in listed() if c["kind"] != "batch")
    for _ in range(1000):
        signal = rng.choice(["toy", "bbh", "bbh", "bbh", "bns"])
        kind = rng.choice(["lnl", "lnl", "nuts", "nuts", "stage"])
        c = dict(kind=kind, signal=signal)
        if signal == "toy":
            c.update(seconds=rng.randint(2, 8), fmax=rng.choice([128, 256]))
        elif signal == "bbh":
            c.update(seconds=_loguniform(rng, 4, 32), fmax=rng.choice([512, 1024, 2048]))
        else:
            c.update(seconds=rng.randint(64, 128), fmax=rng.choice([1024, 2048]))
        c.update(n=_loguniform(rng, 128, 16384))
        if kind == "lnl":
            c.update(where=rng.choice(["prior", "ball"]), precision=rng.choice(["mixed", "mixed", "split", "fp64"]),
                     how=rng.choice(["grad", "grad", "forward", "autograd"]))
        elif kind == "nuts":
            c.update(metric=rng.choice(["identity", "covariance", "local"]), depth=rng.randint(4, 8),
                     precision=rng.choice(["mixed", "mixed", "split", "fp64"]))
            c.update(rng.choice([dict(where="prior", beta=1e-4), dict(where="ball", beta=1.0)]))
        else:
            c.update(beta=rng.choice([0.0, 0.001, 0.03]), metric=rng.choice(["covariance", "local"]))
        if signal == "bns" and kind != "lnl":
            continue  # mutations of the 128 s signal take longer than any listed case
        cost = work(c)["flops"] * (12 if c.get("precision") == "fp64" else 1)
        if cost <= most:
            return c
    raise RuntimeError("no case drawn")


# ------------------------------------------------------------- their workloads


def _workload(case):
    if case["signal"] == "toy":
        w = inputs.tiny()
    elif case["signal"] == "bbh":
        w = inputs.bbh11()
    else:
        w = inputs.bns()
    w.df = 1.0 / case["seconds"]
    w.n_bins = (case["fmax"] - int(w.f_min)) * case["seconds"] + 1
    w.n_particles = case.get("n", w.n_particles)
    w.max_depth = case.get("depth", w.max_depth)
    return w


def _batch_workloads(case):
    every = inputs.batch64()
    return [every[i * len(every) // case["events"]] for i in range(case["events"])]


def _active(w):
    """Bins below the cut-off of the box's middle masses."""
    box = dict(zip(w.phys, zip(w.lo, w.hi)))
    mc, q = sum(box[inputs.MC]) / 2, sum(box[inputs.Q]) / 2
    m = mc * (1 + q) ** 1.2 / q ** 0.6
    cut = 1.0 / (6 ** 1.5 * math.pi * TSUN * m)
    return max(1.0, min(w.n_bins, (cut - w.f_min) / w.df))


def work(case):
    """Evaluations x active bins x detectors: phase (8 terms shared by the detectors), carrier, 20 moment sums."""
    def event(w, evals, grad=True):
        per = 16.0 + w.n_det * (20.0 + (40.0 if grad else 2.0))
        tables = w.n_bins * (9 * 8 + w.n_det * (16 + 8))
        return evals * _active(w) * per, tables

    if case["kind"] == "batch":
        fl = by = 0.0
        for w in _batch_workloads(case):  # some seven stages; trees a quarter of the limit
            f, t = event(w, 7 * w.n_mut * w.n_particles * 2.0 ** (w.max_depth - 2))
            fl, by = fl + f, by + t + w.n_particles * (w.n_dim + 1) * 8
        return {"bytes": by, "flops": fl}
    w = _workload(case)
    n, d = case["n"], w.n_dim
    state = n * (2 * d + 1) * 8.0
    if case["kind"] == "lnl":
        f, t = event(w, n, case["how"] != "forward")
        if case["how"] == "autograd":
            f += event(w, n, False)[0]
        return {"bytes": t + n * 8.0 * (d + 1 + (d if case["how"] != "forward" else 0)), "flops": f}
    if case["kind"] == "nuts":  # two transitions; half the depth limit's leaves
        f, t = event(w, 2 * n * 2.0 ** (case["depth"] - 1))
        return {"bytes": t + 2 * state + n * 32.0 + (2 * n * d * d * 8.0 if case["metric"] == "local" else 0), "flops": f}
    if case["kind"] == "stage":
        f, by = n * (8 * 20.0 + 3.0 * d * d), 2 * state + n * 4.0
        if case["metric"] == "local":  # detectors x (D P2 D products), Cholesky, inverse, Cholesky
            f += n * (w.n_det * (11 * 10 * 10 * 2 + 66 * 10 * 2) + 2.0 * d ** 3)
            by += 2 * n * d * d * 8.0 + w.n_det * 54 * 8.0 * min(n, _active(w))
        return {"bytes": by, "flops": f}
    f, t = event(w, 7 * w.n_mut * n * 2.0 ** (w.max_depth - 2))
    return {"bytes": t + 7 * n * (d + 1) * 8.0, "flops": f}


# ------------------------------------------------ the signal in plain torch, 64 bits


def _detector(det):
    """Arms' tensor (flat 9) and position in light seconds of an L-shaped detector on a sphere."""
    sl, cl, so, co = math.sin(det["lat"]), math.cos(det["lat"]), math.sin(det["lon"]), math.cos(det["lon"])
    east, north = np.array([-so, co, 0.0]), np.array([-sl * co, -sl * so, cl])
    ca, sa = math.cos(det["azimuth"]), math.sin(det["azimuth"])
    x, y = ca * north + sa * east, -sa * north + ca * east
    return 0.5 * (np.outer(x, x) - np.outer(y, y)), EARTH_S * np.array([cl * co, cl * so, sl])


def _physical(w, th):
    cols = [torch.full_like(th[:, 0], v) for v in w.fixed]
    for i, p in enumerate(w.phys):
        cols[p] = th[:, i]
    return cols


def _cutoff(w, th):
    p = _physical(w, th)
    eta = p[inputs.Q] / (1 + p[inputs.Q]) ** 2
    return 1.0 / (6 ** 1.5 * math.pi * TSUN * p[inputs.MC] * eta ** -0.6)


def _response(w, p, dets):
    """Complex response (re, im) [n, det] and delays [n, det]."""
    hp, hx = 0.5 * (1 + p[inputs.COSI] ** 2), p[inputs.COSI]
    re, im, dt = [], [], []
    for det in dets:
        if det.get("fixed_response"):
            fp, fx = det["fplus"] + 0 * hp, det["fcross"] + 0 * hp
            delay = det["delay"] + 0 * hp
        else:
            D, r = _detector(det)
            sa, ca, z = torch.sin(p[inputs.RA]), torch.cos(p[inputs.RA]), p[inputs.SINDEC]
            cd = torch.sqrt(1 - z * z)
            a, b = [sa, -ca, 0 * sa], [z * ca, z * sa, -cd]
            form = lambda u, v: sum(u[i] * float(D[i, j]) * v[j] for i in range(3) for j in range(3))  # noqa: E731
            f0, c0 = form(a, a) - form(b, b), 2 * form(a, b)
            c2, s2 = torch.cos(2 * p[inputs.PSI]), torch.sin(2 * p[inputs.PSI])
            fp, fx = c2 * f0 + s2 * c0, -s2 * f0 + c2 * c0
            delay = -(float(r[0]) * cd * ca + float(r[1]) * cd * sa + float(r[2]) * z)
        re.append(fp * hp)
        im.append(-fx * hx)
        dt.append(delay)
    return torch.stack(re, 1), torch.stack(im, 1), torch.stack(dt, 1)


def _strain(w, th, f, dets):
    """Re and Im of h_a(f_k), [n, det, bins], zero above the cut-off: aligned-spin TaylorF2 to 3.5PN."""
    p = _physical(w, th)
    mc, q, c1, c2 = (p[i][:, None] for i in (inputs.MC, inputs.Q, inputs.CHI1, inputs.CHI2))
    eta, delta = q / (1 + q) ** 2, (1 - q) / (1 + q)
    m1, m2 = 1 / (1 + q), q / (1 + q)
    s, a = 0.5 * (c1 + c2), 0.5 * (c1 - c2)
    beta = (113 / 12 - 19 / 3 * eta) * s + 113 / 12 * delta * a
    gam = (732985 / 2268 - 24260 / 81 * eta - 340 / 9 * eta ** 2) * s + (732985 / 2268 + 140 / 9 * eta) * delta * a
    sig = 79 / 8 * eta * c1 * c2 + 81 / 16 * ((m1 * c1) ** 2 + (m2 * c2) ** 2)
    pi = math.pi
    p2 = 3715 / 756 + 55 / 9 * eta
    p3 = -16 * pi + 4 * beta
    p4 = 15293365 / 508032 + 27145 / 504 * eta + 3085 / 72 * eta ** 2 - 10 * sig
    p5 = pi * (38645 / 756 - 65 / 9 * eta) - gam
    p6 = (11583231236531 / 4694215680 - 640 / 3 * pi ** 2 - 6848 / 21 * 0.57721566490153286061
          + (2255 / 12 * pi ** 2 - 15737765635 / 3048192) * eta + 76055 / 1728 * eta ** 2 - 127825 / 1296 * eta ** 3)
    p7 = pi * (77096675 / 254016 + 378515 / 1512 * eta - 74045 / 756 * eta ** 2)
    u = (pi * TSUN * mc * eta ** -0.6) ** (1 / 3)
    v = u * (f ** (1 / 3))[None, :]
    lv = torch.log(v)
    turns = 3 / (256 * pi * eta) * (v ** -5 + p2 * v ** -3 + p3 * v ** -2 + p4 / v + p5 * (1 + 3 * (lv + 0.5 * math.log(6)))
                                    + (p6 - 6848 / 21 * (lv + math.log(4))) * v + p7 * v ** 2)
    turns = turns - p[inputs.PHIC][:, None] / (2 * pi) - 0.125
    re, im, dt = _response(w, p, dets)
    t = turns[:, None, :] + (p[inputs.TC][:, None] + dt)[:, :, None] * f
    t = 2 * pi * (t - torch.round(t).detach())
    amp = math.sqrt(5 / 24) * pi ** (-2 / 3) * (TSUN * p[inputs.MC]) ** (5 / 6) / (p[inputs.DL] * MPC_S)
    amp = amp[:, None] * (f ** (-7 / 6))[None, :] * (f[None, :] <= _cutoff(w, th)[:, None])
    c, d = torch.cos(t), torch.sin(t)
    return amp[:, None] * (re[..., None] * c + im[..., None] * d), amp[:, None] * (im[..., None] * c - re[..., None] * d)


class _Event:
    """One synthetic event: noise and an injection of the target SNR, from the seed."""

    def __init__(self, w, seed):
        self.w, self.dets, self.psd = w, inputs.detectors(w, seed), inputs.psd_array(w)
        self.f = torch.tensor(inputs.frequencies(w), dtype=torch.float64, device=DEV)
        self.wt = torch.tensor(4 * w.df / self.psd, dtype=torch.float64, device=DEV)
        th = inputs.injection(w, seed)
        k = inputs.distance_index(w)
        if w.snr_target is not None and k is not None:
            hr, hi = self.strain(th)
            rho = math.sqrt(float((self.wt * (hr ** 2 + hi ** 2)).sum()))
            th[k] = min(max(th[k] * rho / w.snr_target, w.lo[k]), w.hi[k])
        hr, hi = self.strain(th)
        self.injection = th
        self.data = torch.stack([hr, hi], -1).cpu().numpy() + inputs.noise(w, seed)
        d = torch.tensor(self.data, device=DEV)
        self.dr, self.di = d[..., 0].contiguous(), d[..., 1].contiguous()
        self.dd = float((self.wt * (self.dr ** 2 + self.di ** 2)).sum())

    def strain(self, th):
        hr, hi = _strain(self.w, torch.tensor(th, device=DEV)[None], self.f, self.dets)
        return hr[0], hi[0]

    def context(self):
        ctx = api.Context.from_workload(self.w)
        ctx.set_data(self.data, self.psd, self.w.f_min, self.w.df, self.dets)
        return ctx

    def theta(self, where, n, seed):
        """Prior draws, or a Gaussian ball around the injection (`where` = its width in prior widths) mirrored into the box."""
        if where == "prior":
            th = inputs.prior_draws(self.w, n, seed)
        else:
            lo, hi = np.array(self.w.lo), np.array(self.w.hi)
            z = np.random.Generator(np.random.Philox(3000 + seed)).standard_normal((n, len(lo)))
            x = np.abs((self.injection - lo) / (hi - lo) + where * z)
            th = lo + np.minimum(x, 2.0 - x) * (hi - lo)
        return torch.tensor(th, dtype=torch.float64, device=DEV)

    def chunks(self, th, cells):
        """Row blocks of th and the number of bins below their cut-off."""
        at = 0
        top = int((self.f <= _cutoff(self.w, th).max()).sum())
        rows = max(1, int(cells / (max(top, 1) * self.w.n_det)))
        while at < len(th):
            yield slice(at, at + rows), max(top, 1)
            at += rows

    def lnl(self, th, grad=True):
        """ln L and its gradient by automatic differentiation."""
        out, g = torch.empty(len(th), dtype=torch.float64, device=DEV), torch.empty_like(th)
        for rows, k in self.chunks(th, 8e6):
            x = th[rows].clone().requires_grad_(grad)
            hr, hi = _strain(self.w, x, self.f[:k], self.dets)
            r = self.wt[:, :k] * (hr * (self.dr[:, :k] - 0.5 * hr) + hi * (self.di[:, :k] - 0.5 * hi))
            v = r.sum((1, 2))
            if grad:
                g[rows] = torch.autograd.grad(v.sum(), x)[0]
            out[rows] = v.detach() - 0.5 * self.dd
        return out, g

    def mass(self, th, beta):
        """beta x Fisher information + prior Hessian + 12 / width^2."""
        n, d = th.shape
        out = torch.empty((n, d, d), dtype=torch.float64, device=DEV)
        for rows, k in self.chunks(th, 2e6):
            x = th[rows]
            cols = []
            for j in range(d):
                e = torch.zeros_like(x)
                e[:, j] = 1
                _, t = torch.func.jvp(lambda y: _strain(self.w, y, self.f[:k], self.dets), (x,), (e,))
                cols.append((torch.stack(t) * torch.sqrt(self.wt[:, :k])).permute(1, 0, 2, 3).reshape(len(x), -1))
            J = torch.stack(cols, 1)
            out[rows] = beta * (J @ J.transpose(1, 2))
        for j in range(d):
            out[:, j, j] += 12 / (self.w.hi[j] - self.w.lo[j]) ** 2
            if self.w.prior[j] == inputs.PRIOR_POWER2:
                out[:, j, j] += 2 / th[:, j] ** 2
        return out


def _inputs(case, seed):
    ev = _Event(_workload(case), seed)
    if case["kind"] == "stage":  # an ensemble part of the way: prior draws, or a wide ball once beta has grown
        th = ev.theta("prior" if case["beta"] == 0 else 0.02, case["n"], seed + 1)
    else:
        th = ev.theta("prior" if case["where"] == "prior" else 1e-3, case["n"], seed + 1)
    return ev, th


# ---------------------------------------------------------------- prepare and run


def _rows(t, n):
    """t in an array of n rows, zeros after it: a run's own number of stages and kept draws differs from event to event."""
    out = t.new_zeros((n,) + tuple(t.shape[1:]))
    out[:len(t)] = t
    return out


def prepare(case, seed):
    s = dict(case)
    if case["kind"] == "batch":
        evs = [_Event(w, seed + i) for i, w in enumerate(_batch_workloads(case))]
        s["batch"] = api.Batch([e.context() for e in evs], [e.w.n_particles for e in evs], evs[0].w.alpha, evs[0].w.n_mut,
                               case["depth"], inputs.METRIC_IDENTITY, evs[0].w.eps_scale, case["precision"])
        s["keys"] = [1000 * seed + i for i in range(len(evs))]
        return s
    if case["kind"] == "run":
        ev = _Event(_workload(case), seed)
        s.update(w=ev.w, ctx=ev.context(), key=1000 + seed)
        return s
    ev, th = _inputs(case, seed)
    s.update(w=ev.w, ctx=ev.context(), theta=th, key=77 + seed)
    if case["kind"] != "lnl":
        s["lnl"], s["grad"] = ev.lnl(th)
    if case["kind"] == "nuts":
        s["cov"] = torch.cov(th.T).contiguous()
    if case["kind"] == "stage":
        s["u"] = float(np.random.Generator(np.random.Philox(seed)).uniform())
    return s


def run(s):
    if s["kind"] == "lnl":
        if s["how"] == "autograd":
            th = s["theta"].clone().requires_grad_(True)
            lnl = api.loglike(th, s["ctx"], s["precision"])
            lnl.sum().backward()
            return {"lnl": lnl.detach(), "grad": th.grad}
        lnl, g = s["ctx"].loglike_grad(s["theta"], s["precision"], grad=s["how"] == "grad")
        return {"lnl": lnl} if g is None else {"lnl": lnl, "grad": g}
    if s["kind"] == "nuts":  # the calls work in place: the ensemble before the stage is kept, as for its pool
        th, lnl, g = s["theta"].clone(), s["lnl"].clone(), s["grad"].clone()
        ctx, w = s["ctx"], s["w"]
        tail = (s["depth"], w.n_mut, s["key"], 256)
        if s["metric"] == "identity":
            st = ctx.nuts_mutate_cov_step(s["beta"], th, lnl, g, s["cov"], w.eps_scale, *tail, precision=s["precision"])
        elif s["metric"] == "covariance":
            st = ctx.nuts_mutate(s["beta"], th, lnl, g, s["cov"], w.eps_scale, *tail, precision=s["precision"])
        else:
            m = ctx.local_metric(th, s["beta"], want=("inv_mass", "chol"))
            st = ctx.nuts_mutate_local(s["beta"], th, lnl, g, m["inv_mass"], m["chol"], w.eps_scale, *tail,
                                       precision=s["precision"])
        return {"theta": th, "lnl": lnl, "grad": g, "accept_and_bins": st.view(torch.float64).view(-1, 4)[:, :2],
                "depth_leapfrogs_divergent": st.view(torch.int32).view(-1, 8)[:, 4:7]}
    if s["kind"] == "stage":
        th, lnl, g = s["theta"].clone(), s["lnl"].clone(), s["grad"].clone()
        r = s["ctx"].reweight_resample(th, lnl, g, s["beta"], s["w"].alpha, s["u"])
        r.update(theta=th, lnl=lnl, grad=g)
        if s["metric"] == "local":
            r.update(s["ctx"].local_metric(th, float(r["beta_next"])))
        return r
    if s["kind"] == "run":
        w, stages = s["w"], 16
        lnz, th, lnl, rec, pth, pll = s["ctx"].smc_run(s["n"], w.alpha, w.n_mut, s["depth"], inputs.METRIC_IDENTITY,
                                                       w.eps_scale, s["key"], s["precision"], pool_stages=stages)
        log_w, kept = api.recycle_run(pth, pll, rec, s["n"], s["key"])
        fields = ("beta", "ess", "dlnz", "eps", "lnz", "accept_mean")
        return {"lnz": np.array(lnz), "theta": th, "lnl": lnl, "pool": _rows(pth, stages * s["n"]),
                "pool_lnl": _rows(pll, stages * s["n"]), "log_w": _rows(log_w, stages * s["n"]),
                "kept": _rows(kept, stages * s["n"]), "n_kept": len(kept),
                "stages": _rows(torch.tensor([[r[k] for k in fields] for r in rec], dtype=torch.float64), stages),
                "leapfrogs": _rows(torch.tensor([r["n_leapfrog"] for r in rec]), stages)}
    res, rounds = s["batch"].run(s["keys"])
    parts = [s["batch"].particles(e) for e in range(len(res))]
    return {"lnz": np.array([r["lnz"] for r in res]), "rounds": rounds, "theta": [p[0] for p in parts],
            "lnl": [p[1] for p in parts]}


# ------------------------------------------------------------------ what they should give


def _stage_exact(case, seed):
    ev, th = _inputs(case, seed)
    lnl, g = ev.lnl(th)
    u = float(np.random.Generator(np.random.Philox(seed)).uniform())
    n, w = len(th), ev.w
    l = lnl.cpu().numpy()
    x = l - l.max()
    ess = lambda b: np.exp(b * x).sum() ** 2 / np.exp(2 * b * x).sum()  # noqa: E731
    lo, hi = 0.0, 1.0 - case["beta"]
    if ess(hi) >= w.alpha * n:
        lo = hi
    else:
        for _ in range(100):
            mid = 0.5 * (lo + hi)
            lo, hi = (mid, hi) if ess(mid) >= w.alpha * n else (lo, mid)
    wt = np.exp(lo * x)
    q = np.cumsum(np.floor(wt * 2.0 ** 32).astype(np.uint64)).astype(object)
    total, U = int(q[-1]), int(math.floor(u * 2.0 ** 32))
    points = [((m << 32) + U) * total // (n << 32) for m in range(n)]
    anc = np.searchsorted(np.array(q, dtype=np.uint64), np.array(points, dtype=np.uint64), side="right")
    a = torch.tensor(anc, device=DEV)
    p = torch.tensor(wt / wt.sum(), device=DEV)
    c = th - (p[:, None] * th).sum(0)
    r = {"beta_next": np.array(case["beta"] + lo), "dlnz": np.array(lo * l.max() + math.log(wt.sum()) - math.log(n)),
         "ess": np.array(wt.sum() ** 2 / (wt ** 2).sum()), "ancestors": torch.tensor(anc.astype(np.int32)),
         "cov": c.T @ (p[:, None] * c), "theta": th[a], "lnl": lnl[a], "grad": g[a]}
    if case["metric"] == "local":
        r["mass"] = ev.mass(r["theta"], float(r["beta_next"]))
        r["inv_mass"] = torch.linalg.inv(r["mass"])
        r["chol"] = torch.linalg.cholesky(0.5 * (r["inv_mass"] + r["inv_mass"].transpose(1, 2)))
    return r


def exact(case, seed):
    """Likelihoods and stages in 64 bits; a NUTS trajectory (kinds nuts, run, batch) has no value but the code's own."""
    if case["kind"] == "stage":
        return _stage_exact(case, seed)
    if case["kind"] != "lnl":
        return None
    ev, th = _inputs(case, seed)
    lnl, g = ev.lnl(th, case["how"] != "forward")
    return {"lnl": lnl} if case["how"] == "forward" else {"lnl": lnl, "grad": g}
