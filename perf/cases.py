"""The calls that users of this library make, with inputs drawn from a seed, for measuring it.

A case is one call through the public Python entry points: a single solve, a batched solve, a
two-grid solve, the differentiable misfit forward and backward, the host-buffer misfit step, or
the least-squares misfit.  Gathers are receivers x time samples, float32; their events are those
of the seeded generators of the tests and the benchmark (hyperbolas, reflections, transmitted
events, a shifted wavelet), evaluated on the GPU.
"""

from __future__ import annotations

import math

import numpy as np
import torch

import paper_1808_07284_gb300 as emd

ISO = emd.EMD_NORM_ISO


def listed():
    return [
        # The least-squares misfit of one small gather and its gradient: the conventional step
        # that the transport misfit is compared with, and the smallest call there is.
        {"name": "lsd_256x64", "op": "lsd", "kind": "hyperbolic", "nr": 64, "nt": 256, "batch": 1,
         "dt": 2e-3, "dx": 10.0},
        # The one-dimensional time-shift study: 61 shifts of one trace in one batched call.
        {"name": "sweep_61x1x1024", "op": "batch", "kind": "wavelet", "nr": 1, "nt": 1024, "batch": 61,
         "dt": 1.0 / 1023, "dx": 1.0, "iters": 100},
        # The small single gather of the tests, solved alone: launches and latency.
        {"name": "solve_256x64", "op": "solve", "kind": "hyperbolic", "nr": 64, "nt": 256, "batch": 1,
         "dt": 2e-3, "dx": 10.0, "iters": 200},
        # A crosshole gather on the unit square, 100 iterations, with the isotropic ground cost.
        {"name": "solve_1000x128_iso", "op": "solve", "kind": "transmissive", "nr": 128, "nt": 1000,
         "batch": 1, "dt": 1.0 / 999, "dx": 1.0 / 127, "iters": 100, "iso": True},
        # A resampled streamer gather on its transport grid, 200 iterations.
        {"name": "solve_401x321", "op": "solve", "kind": "reflective", "nr": 321, "nt": 401, "batch": 1,
         "dt": 1e-2, "dx": 25.0, "iters": 200},
        # The transmissive gather of the benchmark, solved alone.
        {"name": "solve_3000x400", "op": "solve", "kind": "transmissive", "nr": 400, "nt": 3000, "batch": 1,
         "dt": 1e-3, "dx": 12.5, "iters": 100},
        # The same gather by the two-grid solve: 150 coarse iterations, then a short fine solve.
        {"name": "two_grid_3000x400", "op": "two_grid", "kind": "transmissive", "nr": 400, "nt": 3000,
         "batch": 1, "dt": 1e-3, "dx": 12.5, "iters": 20, "factor": 10, "coarse": 150},
        # Shots of uneven sizes in one batched solve with a stopping residual, capped at 80
        # iterations (the cap is what ends it, as in the paper's runs).
        {"name": "uneven_12", "op": "batch", "kind": "hyperbolic", "nr": 0, "nt": 0, "batch": 12,
         "dt": 1e-3, "dx": 12.5, "iters": 80, "tol": 1e-4},
        # The differentiable misfit of 16 reflective gathers: forward and backward.
        {"name": "grad_16x4000x480", "op": "grad", "kind": "reflective", "nr": 480, "nt": 4000, "batch": 16,
         "dt": 1e-3, "dx": 12.5, "iters": 80},
        # The misfit step of an inversion whose gathers are in host memory.
        {"name": "host_4x4000x480", "op": "host", "kind": "reflective", "nr": 480, "nt": 4000, "batch": 4,
         "dt": 1e-3, "dx": 12.5, "iters": 80},
        # One marine-streamer shot, solved alone.
        {"name": "solve_8000x648", "op": "solve", "kind": "marine", "nr": 648, "nt": 8000, "batch": 1,
         "dt": 2e-3, "dx": 25.0, "iters": 100},
        # Marine-streamer shots in one batched solve, the benchmark's flagship in small.
        {"name": "batch_16x8000x648", "op": "batch", "kind": "marine", "nr": 648, "nt": 8000, "batch": 16,
         "dt": 2e-3, "dx": 25.0, "iters": 100},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    op = rng.choice(["lsd", "batch", "batch", "solve", "solve", "solve", "two_grid", "grad", "host"])
    kind = rng.choice(["hyperbolic", "transmissive", "reflective", "marine"])
    case = {"op": op, "kind": kind, "nr": _log_int(rng, 8, 648), "nt": _log_int(rng, 64, 8000), "batch": 1}
    if op == "batch" and rng.random() < 0.25:
        case.update(kind="wavelet", nr=1, nt=_log_int(rng, 64, 4096), batch=rng.randint(2, 61))
    elif op == "batch" and rng.random() < 0.35:
        case.update(nr=0, nt=0, batch=rng.randint(2, 12), kind="hyperbolic")
    elif op in ("batch", "grad"):
        case["batch"] = rng.randint(2, 16)
    elif op == "host":
        case["batch"] = rng.randint(1, 4)
    if op == "two_grid":
        case["factor"] = rng.choice([4, 8, 10])
        case["coarse"] = rng.randint(50, 150)
        case["nt"] = max(case["nt"], 40 * case["factor"])
    if op != "lsd":
        case["iters"] = rng.randint(10, 30) if op == "two_grid" else rng.randint(40, 80)
        if op in ("solve", "batch") and rng.random() < 0.2:
            case["iso"] = True
        if op == "batch" and rng.random() < 0.3:
            case["tol"] = 1e-4
    if case["kind"] == "wavelet":
        case.update(dt=1.0 / (case["nt"] - 1), dx=1.0)
    elif rng.random() < 0.25 and case["nr"] > 1:  # the unit square
        case.update(dt=1.0 / (case["nt"] - 1), dx=1.0 / (case["nr"] - 1))
    else:
        dt, dx = {"hyperbolic": (1e-3, 12.5), "transmissive": (1e-3, 12.5), "reflective": (1e-3, 12.5),
                  "marine": (2e-3, 25.0)}[case["kind"]]
        case.update(dt=dt, dx=dx)
    return case


# ---------------------------------------------------------------------------------- inputs


def _sizes(case):
    """The (receivers, samples) of every gather of a case."""
    if case["nr"]:
        return [(case["nr"], case["nt"])] * case["batch"]
    rng = np.random.default_rng(3 + case["batch"])  # uneven shots: 200..640 x 1500..5000
    nrs = rng.integers(200, 641, case["batch"])
    nts = rng.integers(1500, 5001, case["batch"])
    return [(int(a), int(b)) for a, b in zip(nrs, nts)]


def _events(out, times, tau, amp, f0):
    """out += sum_e amp[e] ricker(t - tau[e]), row by row."""
    for e in range(tau.shape[0]):
        a = ((times[None, :] - tau[e][:, None]) * (math.pi * f0)).square_()
        out += amp[e][:, None] * (1.0 - 2.0 * a) * torch.exp(-a)


def _pair(kind, nr, nt, rng, dev, shift=None):
    """(observed, predicted) on an nr x nt grid.  The events are laid out on a record of 16 s
    (marine), 4 s or as many samples as there are at the generator's own sampling, so that every
    size carries events inside the record."""
    step, dx, f0, n = {"hyperbolic": (1e-3, 12.5, 10.0, 3), "transmissive": (1e-3, 12.5, 8.0, 8),
                       "reflective": (1e-3, 12.5, 6.0, 20), "marine": (2e-3, 25.0, 5.0, 41),
                       "wavelet": (1.0 / (nt - 1), 1.0, 8.0, 1)}[kind]
    if kind != "wavelet" and nt * step < 2.0:  # short records: coarser sampling of the same events
        step = 2.0 / nt
    if kind != "wavelet":
        dx = max(dx, 4800.0 / nr) if nr < 384 else dx
    x = (np.arange(nr) + 1.0) * dx
    end = nt * step
    if kind == "wavelet":
        s = rng.uniform(-0.3, 0.3) if shift is None else shift
        tau_o, tau_p, amp = np.full((1, 1), 0.5), np.full((1, 1), 0.5 + s), np.ones((1, 1))
    elif kind == "transmissive":
        tau = [x / rng.uniform(1500, 2000)]
        tau += [x / rng.uniform(2500, 4500) + rng.uniform(0.1, 0.8) for _ in range(3)]
        tau += [np.sqrt(rng.uniform(0.3, 2.5) ** 2 + (x - rng.uniform(0, nr * dx)) ** 2 / rng.uniform(1800, 3000) ** 2)
                for _ in range(4)]
        tau_o = np.array(tau) * (end / 4.0)
        tau_p = tau_o + rng.uniform(-1.5, 1.5, 8)[:, None] / f0
        amp = rng.uniform(0.2, 1.0, 8)[:, None] * np.sqrt(x[0] / x)[None, :]
    else:
        t0 = np.sort(rng.uniform(0.05, 0.95, n)) * min(end, 4.0 if kind != "marine" else end)
        v = 1500.0 + 400.0 * t0
        tau_o = np.sqrt(t0[:, None] ** 2 + (x[None, :] / v[:, None]) ** 2)
        if kind == "hyperbolic":
            tau_p = np.sqrt((t0 + rng.uniform(-0.04, 0.04, n))[:, None] ** 2 + (x[None, :] / v[:, None]) ** 2)
            amp = np.ones((n, nr))
        else:
            if kind == "marine":
                vp = v * (1.0 + rng.uniform(-0.15, 0.15))
            else:
                vp = v * (1.0 + 0.08 * np.sin(0.5 * math.pi * t0 + rng.uniform(0.0, 2.0 * math.pi)))
            tau_p = np.sqrt(t0[:, None] ** 2 + (x[None, :] / vp[:, None]) ** 2)
            amp = np.repeat(rng.standard_normal(n)[:, None], nr, axis=1)
    times = torch.arange(nt, device=dev, dtype=torch.float32) * step
    obs = torch.zeros((nr, nt), device=dev)
    pred = torch.zeros((nr, nt), device=dev)
    tau_o, tau_p, amp = (torch.from_numpy(np.ascontiguousarray(a, dtype=np.float32)).to(dev) for a in (tau_o, tau_p, amp))
    _events(obs, times, tau_o, amp, f0)
    _events(pred, times, tau_p, amp, f0)
    if kind in ("transmissive", "marine"):  # 30 dB white noise / 20 dB noise of 3-15 Hz
        gen = torch.Generator(device=dev)
        gen.manual_seed(int(rng.integers(1 << 31)))
        noise = torch.randn((nr, nt), device=dev, generator=gen)
        if kind == "marine":
            spec = torch.fft.rfft(noise, dim=1)
            fr = torch.fft.rfftfreq(nt, step, device=dev)
            noise = torch.fft.irfft(spec * ((fr >= 3.0) & (fr <= 15.0)), n=nt, dim=1).contiguous()
        base = pred if kind == "transmissive" else obs
        level = base.square().mean().sqrt() * 10.0 ** (-(30.0 if kind == "transmissive" else 20.0) / 20.0)
        base += noise * (level / noise.square().mean().sqrt().clamp_min(1e-30))
    return obs, pred


def _gathers(case, seed):
    dev = torch.device("cuda", torch.cuda.current_device())
    rng = np.random.default_rng(int(seed))
    pairs = []
    for b, (nr, nt) in enumerate(_sizes(case)):
        shift = None
        if case["kind"] == "wavelet":  # the sweep's shifts, moved as a whole by the seed
            shift = -0.3 + 0.6 * (b + rng.uniform(0.1, 0.9)) / case["batch"]
        pairs.append(_pair(case["kind"], nr, nt, rng, dev, shift))
    weights = torch.from_numpy(rng.uniform(0.5, 1.5, case["batch"]).astype(np.float32)).to(dev)
    return [p[0] for p in pairs], [p[1] for p in pairs], weights


def prepare(case, seed):
    obs, pred, weights = _gathers(case, seed)
    s = {"op": case["op"], "obs": obs, "pred": pred, "dt": case["dt"], "dx": case["dx"]}
    kw = {}
    if "iters" in case:
        kw["max_iter"] = case["iters"]
    if case.get("iso"):
        kw["norm"] = ISO
    if case.get("tol"):
        kw["tol"] = case["tol"]
    s["kw"] = kw
    dev = obs[0].device
    nts, nrs = [int(t.shape[1]) for t in obs], [int(t.shape[0]) for t in obs]
    if case["op"] == "solve":
        s["ws"] = emd.new_workspace(emd.emd_workspace_size(nts[0], nrs[0]), dev)
    elif case["op"] == "two_grid":
        s["grid"] = {"factor": case["factor"], "coarse_max_iter": case["coarse"]}
        s["ws"] = emd.new_workspace(emd.emd_mg_workspace_size(nts[0], nrs[0], case["factor"]), dev)
    elif case["op"] == "batch":
        s["ws"] = emd.new_workspace(emd.emd_batched_workspace_size(nts, nrs), dev)
        if case["nr"]:  # equal sizes: one array of potentials and one of fluxes, a view for each shot
            s["phi"] = torch.empty((len(obs), nrs[0], nts[0]), device=dev)
            s["m"] = torch.empty((len(obs), 2, nrs[0], nts[0]), device=dev)
            s["params"] = emd.emd_default_params(**kw)
    elif case["op"] == "grad":
        s["pred"] = [p.requires_grad_(True) for p in pred]
        s["weights"] = weights
    elif case["op"] == "lsd":
        s["pred"] = [pred[0].requires_grad_(True)]
    elif case["op"] == "host":
        s["obs"] = [o.cpu().pin_memory() for o in obs]
        s["pred"] = [p.cpu().pin_memory() for p in pred]
        s["grads"] = [torch.empty(tuple(o.shape)).pin_memory() for o in obs]
        s["ws"] = emd.new_workspace(emd.emd_misfit_batched_host_workspace_size(nts, nrs), dev)
    return s


def run(s):
    op, obs, pred, dt, dx, kw = s["op"], s["obs"], s["pred"], s["dt"], s["dx"], s["kw"]
    if op == "solve":
        dist, phi, m, _ = emd.emd(obs[0], pred[0], dt, dx, workspace=s["ws"], **kw)
        return {"dist": dist, "phi": phi, "m": m}
    if op == "two_grid":
        dist, phi, m, _ = emd.emd(obs[0], pred[0], dt, dx, workspace=s["ws"], multigrid=s["grid"], **kw)
        return {"dist": dist, "phi": phi, "m": m}
    if op == "batch":
        if "phi" in s:
            B = len(obs)
            res = emd.emd_dyn_solve_batched(obs, pred, [dt] * B, [dx] * B, s["params"], list(s["phi"].unbind(0)),
                                            list(s["m"].unbind(0)), s["ws"])
            return {"dist": np.array([r.dist for r in res], dtype=np.float32), "phi": s["phi"], "m": s["m"]}
        dists, phis, ms, _ = emd.emd_batched(obs, pred, dt, dx, workspace=s["ws"], **kw)
        return {"dist": np.array(dists, dtype=np.float32), "phi": phis, "m": ms}
    if op == "grad":
        loss = emd.emd_loss_batched(pred, obs, dt, dx, **kw)
        grads = torch.autograd.grad((loss * s["weights"]).sum(), pred)
        return {"loss": loss.detach(), "grad": list(grads)}
    if op == "host":
        dists, grads, _ = emd.emd_misfit_host(obs, pred, dt, dx, grad_preds=s["grads"], workspace=s["ws"], **kw)
        return {"dist": np.array(dists, dtype=np.float32), "grad": grads}
    loss = emd.lsd_loss(pred[0], obs[0], dt, dx)
    (grad,) = torch.autograd.grad(loss, pred[0])
    return {"loss": loss.detach(), "grad": grad}


def work(case):
    """Bytes: both gathers read, and every output written, once.  Flops: about 45 per cell and
    PDHG iteration (prox 14, divergences 10, dual step 4, linesearch sums 17)."""
    cells = sum(nr * nt for nr, nt in _sizes(case))
    if case["op"] == "lsd":
        return {"bytes": 12.0 * cells, "flops": 4.0 * cells}
    out = 4.0 if case["op"] in ("grad", "host") else 12.0
    flops = 45.0 * cells * case["iters"]
    if case["op"] == "two_grid":
        nc = -(-case["nt"] // case["factor"])
        flops += 45.0 * case["nr"] * nc * case["coarse"] + 3.0 * 2.0 * cells * nc
    return {"bytes": (8.0 + out) * cells, "flops": flops}


# ------------------------------------------------------------------------- in 64 bits


def _solve64(obs, pred, dt, dx, iters, iso=False, phi=None, u=None, eps=1e-4, zeta=0.99, delta=1e5):
    """PDHG with linesearch (Algorithm 1) in float64: (dist, phi, [ux, ut])."""
    f = pred.double() - obs.double()
    f -= f.mean()
    nr, nt = f.shape
    one = nr == 1
    rx, rt = (0.0 if one else 1.0 / dx), 1.0 / dt
    lam = 4.0 * rt * rt + 4.0 * rx * rx

    def grad(a):
        gx, gt = torch.zeros_like(a), torch.zeros_like(a)
        gx[1:] = (a[1:] - a[:-1]) * rx
        gt[:, 1:] = (a[:, 1:] - a[:, :-1]) * rt
        return gx, gt

    def div(x, t):
        d = torch.zeros_like(x)
        d[:-1] += x[1:] * rx
        d[1:] -= x[1:] * rx
        d[:, :-1] += t[:, 1:] * rt
        d[:, 1:] -= t[:, 1:] * rt
        return d

    phi = torch.zeros_like(f) if phi is None else phi.clone()
    ux, ut = (torch.zeros_like(f), torch.zeros_like(f)) if u is None else (u[0].clone(), u[1].clone())
    ux[0], ut[:, 0] = 0.0, 0.0
    alpha, theta = 1.0 / math.sqrt(delta * lam), 1.0
    for _ in range(iters):
        gx, gt = grad(phi)
        vx, vt = ux + alpha * gx, ut + alpha * gt
        if iso:
            n = (vx * vx + vt * vt).sqrt()
            s = torch.where(n > alpha, 1.0 - alpha / n.clamp_min(1e-300), torch.zeros_like(n)) / (1.0 + eps * alpha)
            nx, nv = s * vx, s * vt
        else:
            nx = (vx - vx.clamp(-alpha, alpha)) / (1.0 + eps * alpha)
            nv = (vt - vt.clamp(-alpha, alpha)) / (1.0 + eps * alpha)
        p, q = div(nx, nv) + f, div(nx - ux, nv - ut)
        (px, pt), (qx, qt) = grad(p), grad(q)
        sums = torch.stack([(p * p).sum(), (p * q).sum(), (q * q).sum(), (px * px).sum() + (pt * pt).sum(),
                            (px * qx).sum() + (pt * qt).sum(), (qx * qx).sum() + (qt * qt).sum()]).tolist()
        s = math.sqrt(1.0 + theta)
        for _trial in range(40):
            a = alpha * s
            if delta * a * a * (sums[3] + 2 * s * sums[4] + s * s * sums[5]) <= zeta * zeta * (
                    sums[0] + 2 * s * sums[1] + s * s * sums[2]):
                break
            s *= 0.5
        alpha, theta = alpha * s, s
        phi += delta * alpha * (p + theta * q)
        ux, ut = nx, nv
    norm = (ux * ux + ut * ut).sqrt().sum() if iso else ux.abs().sum() + ut.abs().sum()
    area = dt if one else dx * dt
    return area * float(norm + 0.5 * eps * ((ux * ux).sum() + (ut * ut).sum())), phi, [ux, ut]


def _sinc64(a, r, nt, staggered):
    n = torch.arange(nt, device=a.device, dtype=torch.float64)
    x = n / r if staggered else (n - (r - 1) / 2.0) / r
    return a @ torch.sinc(x[None, :] - torch.arange(a.shape[1], device=a.device, dtype=torch.float64)[:, None])


def exact(case, seed):
    obs, pred, weights = _gathers(case, seed)
    dt, dx = case["dt"], case["dx"]
    if case["op"] == "lsd":
        d = pred[0].double() - obs[0].double()
        area = dt if case["nr"] == 1 else dx * dt
        return {"loss": 0.5 * area * d.square().sum(), "grad": area * d}
    if sum(o.numel() for o in obs) * case["iters"] > 5e9 or len(obs) * case["iters"] > 20000:
        return None
    iso = bool(case.get("iso"))
    dists, phis, ms = [], [], []
    for o, p in zip(obs, pred):
        phi = u = None
        if case["op"] == "two_grid":
            r, nt = case["factor"], case["nt"]
            pad = (-nt) % r
            oc, pc = (torch.nn.functional.pad(a.double(), (0, pad)).reshape(a.shape[0], -1, r).mean(2) for a in (o, p))
            _, cphi, cu = _solve64(oc, pc, dt * r, dx, case["coarse"], iso)
            phi = _sinc64(cphi, r, nt, False)
            u = [_sinc64(cu[0], r, nt, False), _sinc64(cu[1], r, nt, True)]
        dist, phi, u = _solve64(o, p, dt, dx, case["iters"], iso, phi, u)
        dists.append(dist)
        phis.append(phi)
        ms.append(torch.stack(u))
    if case["op"] in ("grad", "host"):
        grads = [(dx * dt if o.shape[0] > 1 else dt) * (phi - phi.mean()) for o, phi in zip(obs, phis)]
        if case["op"] == "host":
            return {"dist": np.array(dists), "grad": grads}
        return {"loss": torch.tensor(dists, dtype=torch.float64),
                "grad": [w * g for w, g in zip(weights.double(), grads)]}
    if case["op"] == "batch":
        if case["nr"]:
            return {"dist": np.array(dists), "phi": torch.stack(phis), "m": torch.stack(ms)}
        return {"dist": np.array(dists), "phi": phis, "m": ms}
    return {"dist": dists[0], "phi": phis[0], "m": ms[0]}
