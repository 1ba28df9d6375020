"""Workloads that stand for what a user of gcpush runs, one pass of each through the public API.

Four kinds of work, every one with inputs made from the seed on the GPU:

* ``push``: electrons advanced through a gridded wind (``Context.advance``) and read back, as
  one segment of a long run: small and large ensembles, FP32-mixed and FP64, steady,
  two-fluid and time-dependent fields, wind-frame collisions, tallies, cell sort, graph replay;
* ``neural``: the same with the field taken from a SIREN (the split-step push);
* ``heldout``: the network and its Jacobian, and the grid's interpolant, at test points;
* ``grad`` / ``fit``: the training's loss and gradient on one batch, and a whole short fit.

The wind is the Parker spiral with the solenoidal perturbation of ``synth`` (its modes are
drawn from the seed), sampled on the nodes with torch. A push state is returned as the
library hands it over (18 arrays), so trajectories are compared in full.
"""
import functools
import math

import numpy as np
import torch

from paper_2403_06706_gb300 import gcpush, synth

AU = synth.AU
GRIDS = {"small": (64, 32, 64), "odd": (97, 49, 131), "main": (256, 128, 256), "large": (512, 256, 512)}
N_SIREN = gcpush.SIREN_NPARAMS


def _push(name, **kw):
    case = {"name": name, "kind": "push", "grid": "main", "n": 4096, "ens": 1, "steps": 100, "burn": 0,
            "prec": "f32", "mode": "ideal", "wind_u": 0.0, "mu_law": 0, "scatter_law": 0, "spectrum": False,
            "tally": 0, "sort": 0, "graph": False, "restore": False}
    case.update(kw)
    return case


def listed():
    return [
        # the smallest production call: a few thousand test electrons on the coarse Parker grid
        _push("push32_4096", grid="small", n=4096, steps=400),
        # the plain FP64 workload, as configured: 4096 electrons for 30 min of 0.5 s steps
        _push("push64_4096", grid="small", n=4096, steps=3600, prec="f64"),
        # the benchmark's population and field with its tallies and cell sort: one checkpointed
        # segment (restore from pinned host memory, 1000 steps, read state and tallies back)
        _push("push32_3e6", n=3_000_000, ens=3, steps=1000, burn=500, tally=32, sort=1000, restore=True),
        # 64 uneven ensembles in one context, replayed as a captured graph
        _push("push32_batch64", n=0, ens=64, steps=500, graph=True),
        # the large grid (2.1 GB) with a power-law spectrum and fine tallies
        _push("push32_large", grid="large", n=2_000_003, steps=500, burn=500, spectrum=True, tally=64, sort=1000),
        # a ragged population in a two-fluid field, collisions in the wind frame, Eq. 12's law
        _push("push32_two_fluid", n=200_003, ens=2, steps=500, mode="two_fluid", wind_u=4.0e5, scatter_law=1),
        # a time-dependent field: two snapshots blended over half an hour
        _push("push32_time", n=500_009, ens=2, steps=250, mode="time"),
        # electrons pushed through the neural field: a thousand (tests and studies of the
        # field), and a production-sized population
        {"name": "neural_1024", "kind": "neural", "n": 1024, "steps": 100},
        {"name": "neural_1e6", "kind": "neural", "n": 1_000_003, "steps": 20},
        # field quality on held-out points: grid interpolant, network and Jacobian
        {"name": "heldout_1e6", "kind": "heldout", "n": 1_048_576},
        # one training batch: loss and gradient of 65536 samples
        {"name": "grad_65536", "kind": "grad", "n": 65536},
        # a short fit: 10^6 samples, two epochs of Adam
        {"name": "fit_1e6", "kind": "fit", "n": 1_000_000, "batch": 65536, "epochs": 2},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["push", "push", "push64", "neural", "heldout", "grad", "fit"])
    if kind == "push":
        n = _log(rng, 1000, 3_000_000)
        grid = rng.choice(["small", "odd", "main", "main"])
        mode = rng.choice(["ideal", "ideal", "two_fluid", "time"])
        steps = max(10, min(_log(rng, 20, 1000), 1_000_000_000 // n))
        c = _push("", grid=grid, n=n, ens=rng.choice([1, 2, 3, 7]), steps=steps, mode=mode,
                  wind_u=rng.choice([0.0, 0.0, 4.0e5]), mu_law=rng.choice([0, 0, 1]),
                  scatter_law=rng.choice([0, 1]), spectrum=rng.random() < 0.3, tally=rng.choice([0, 16, 32]),
                  sort=rng.choice([0, 0, 250]), graph=rng.random() < 0.25, restore=rng.random() < 0.25)
        del c["name"]
        return c
    if kind == "push64":
        n = _log(rng, 500, 200_000)
        c = _push("", grid=rng.choice(["small", "odd", "main"]), n=n, ens=rng.choice([1, 3]), prec="f64",
                  steps=max(10, min(_log(rng, 20, 3600), 40_000_000 // n)), mode=rng.choice(["ideal", "two_fluid"]),
                  tally=rng.choice([0, 16]))
        del c["name"]
        return c
    if kind == "neural":
        n = _log(rng, 200, 1_000_000)
        return {"kind": "neural", "n": n, "steps": max(4, min(_log(rng, 4, 100), 20_000_000 // n))}
    if kind == "heldout":
        return {"kind": "heldout", "n": _log(rng, 100, 2_000_000)}
    if kind == "grad":
        return {"kind": "grad", "n": 128 * _log(rng, 1, 2048)}
    batch = 128 * _log(rng, 64, 1024)
    return {"kind": "fit", "n": batch + _log(rng, 50_000, 1_500_000), "batch": batch, "epochs": rng.choice([1, 2])}


# ------------------------------------------------------------------------------- inputs


def _spec(grid, seed, **kw):
    n_r, n_th, n_ph = GRIDS[grid]
    pert = {} if grid == "small" else {"eps": 0.2, "n_modes": 16} if grid == "large" else {"eps": 0.1, "n_modes": 8}
    return synth.WindSpec(n_r, n_th, n_ph, seed=seed, **{**pert, **kw})


def _wind(spec, dtype):
    """The nodes of synth.wind_grid, computed on the GPU."""
    f8 = {"dtype": torch.float64, "device": "cuda"}
    r = (spec.r_min_au + spec.dr_au * torch.arange(spec.n_r, **f8)) * AU
    th = math.pi * torch.arange(spec.n_th, **f8) / (spec.n_th - 1)
    ph = 2.0 * math.pi * torch.arange(spec.n_ph, **f8) / spec.n_ph
    st = torch.sin(th)
    st[0] = st[-1] = 0.0
    out = torch.empty((spec.n_ph, spec.n_th, spec.n_r, 8), dtype=dtype, device="cuda")
    k, e, psi, a = (torch.from_numpy(np.ascontiguousarray(m)).cuda() for m in synth.perturbation_modes(spec))
    w, c = spec.omega / spec.u_sw, spec.B1 * AU * AU
    cross = functools.partial(torch.linalg.cross, dim=-1)
    step = max(1, 4_000_000 // (spec.n_th * spec.n_r))
    for lo in range(0, spec.n_ph, step):
        p = ph[lo:lo + step, None, None]
        rr = r[None, None, :].expand(len(p), spec.n_th, -1)
        x = torch.stack([rr * st[None, :, None] * torch.cos(p), rr * st[None, :, None] * torch.sin(p),
                         (r[None, :] * torch.cos(th)[:, None])[None].expand_as(rr)], -1)
        zxr = torch.stack([-x[..., 1], x[..., 0], torch.zeros_like(rr)], -1)
        b = c * (x / (rr**3)[..., None] - w * zxr / (rr**2)[..., None])
        if spec.n_modes:
            s = torch.sqrt(1.0 + (w * rr) ** 2)
            g = spec.eps * c * s / rr**2
            dg = spec.eps * c * (-2.0 * s / rr**3 + w * w / (rr * s))
            vec, curl = torch.zeros_like(x), torch.zeros_like(x)
            for m in range(spec.n_modes):
                km = torch.linalg.vector_norm(k[m])
                q = x @ k[m] + psi[m]
                vec += (a[m] / km * torch.sin(q))[..., None] * e[m]
                curl += (a[m] * torch.cos(q))[..., None] * cross(k[m] / km, e[m])
            b = b + dg[..., None] * cross(x / rr[..., None], vec) + g[..., None] * curl
        o = out[lo:lo + step]
        o[..., 0:3] = b
        o[..., 3:6] = -spec.u_sw * cross(x / rr[..., None], b)
        o[..., 6] = torch.linalg.vector_norm(b, dim=-1)
        o[..., 7] = spec.phi1_v * (AU / rr) ** (2.0 * (spec.gamma_p - 1.0)) if spec.phi1_v else 0.0
    return out


def _pinned(shape, dt):
    t = torch.empty(shape, dtype=torch.float64 if dt == np.float64 else torch.int32, pin_memory=True)
    return t.numpy().view(dt)


def _ensembles(case, spec):
    if case["ens"] == 64:
        return list(synth.c3_batched().ensembles)
    r_out, ens, left = synth.r_out_default(spec), [], case["n"]
    for k in range(case["ens"]):
        cnt = left // (case["ens"] - k)
        left -= cnt
        law = {"energy_law": 1} if case["spectrum"] else {}
        ens.append(synth.EnsembleSpec(cnt, lam_au=(0.5, 0.1, 1.0, 0.3, 0.7, 0.05, 2.0)[k], lat_deg=24.0 - 7.0 * k,
                                      r_out_au=r_out, mu_law=case["mu_law"], scatter_law=case["scatter_law"], **law))
    return ens


def _prepare_push(case, seed):
    f64 = case["prec"] == "f64"
    dtype = torch.float64 if f64 else torch.float32
    spec = _spec(case["grid"], seed % 65521, phi1_v=200.0 if case["mode"] == "two_fluid" else 0.0)
    ctx = gcpush.Context(precision=gcpush.PREC_FP64 if f64 else gcpush.PREC_FP32_MIXED, seed=seed & 0x7FFFFFFF,
                         wind_u=case["wind_u"])
    ctx.field_load(_wind(spec, dtype), spec.r_min_au, spec.r_max_au, ideal=2 if case["mode"] == "two_fluid" else True)
    if case["mode"] == "time":
        later = _spec(case["grid"], (seed + 1) % 65521, B1=4.2e-9, u_sw=5.0e5)
        ctx.field_load_next(_wind(later, dtype), 0.0, 1800.0)
    ctx.inject(_ensembles(case, spec))
    if case["sort"]:
        ctx.set_launch(sort_every=case["sort"])
    if case["burn"]:
        ctx.advance(0.5, case["burn"])
    if case["tally"]:
        b = case["tally"]
        ctx.tally_arm(cadence=max(1, min(100, case["steps"] // 2)), n_mu=b, n_E=b, n_r=2 * b)
    if case["graph"]:
        ctx.set_graph(True)
    host = gcpush.state_buffers(ctx.n, alloc=_pinned)
    if case["restore"]:
        ctx.get_state(out=host)
    return {"case": case, "ctx": ctx, "host": host}


@functools.lru_cache(maxsize=1)
def _network():
    """Weights of a network that represents the Parker wind to several percent: seeded sine
    layers, and the output layer by least squares on points of the shell (in closed form: a
    fit by Adam would take seconds and is not reproducible bit for bit). omega0 = 10."""
    spec = synth.WindSpec(*GRIDS["main"])
    p = synth.siren_init(0).astype(np.float64)
    rng = np.random.default_rng(1)
    v = rng.normal(size=(12288, 3))
    x = v / np.linalg.norm(v, axis=1, keepdims=True) * rng.uniform(0.1, 1.0, (12288, 1))
    h = np.sin(10.0 * (x @ p[:768].reshape(256, 3).T + p[768:1024]))
    for o in (1024, 66816, 132608):
        h = np.sin(h @ p[o:o + 65536].reshape(256, 256).T + p[o + 65536:o + 65792])
    pos = x * spec.r_max_au * AU
    b, e = synth.wind_at(spec, pos)
    r = np.linalg.norm(pos, axis=1, keepdims=True) / AU
    t = np.concatenate([b * r**2 / spec.B1, e * r / (spec.B1 * spec.u_sw),
                        np.linalg.norm(b, axis=1, keepdims=True) * r**2 / spec.B1, 0 * r], 1)
    h = np.concatenate([h, np.ones((len(h), 1))], 1)
    s = np.linalg.solve(h.T @ h + 1e-3 * np.eye(257), h.T @ t)
    p[198400:200448] = s[:256].T.ravel()
    p[200448:] = s[256]
    return p.astype(np.float32)


def _net_context(seed, params, omega0, grid="main"):
    spec = _spec(grid, seed % 65521)
    nodes = _wind(spec, torch.float32)
    ctx = gcpush.Context(seed=seed & 0x7FFFFFFF)
    ctx.field_load(nodes, spec.r_min_au, spec.r_max_au)
    sc = synth.field_scales(spec)
    desc = {"omega0": omega0, "r_max_au": spec.r_max_au, "B_scale": sc["B_scale"], "E_scale": sc["E_scale"]}
    ctx.siren_set(params, **desc)
    return spec, nodes, ctx, desc


def _points(n, spec, seed):
    """Points uniform in the volume of the grid's shell, scaled by r_max."""
    g = torch.Generator(device="cuda").manual_seed(seed)
    a, b = (spec.r_min_au / spec.r_max_au) ** 3, 1.0
    r = (a + (b - a) * torch.rand((n, 1), generator=g, device="cuda", dtype=torch.float64)) ** (1.0 / 3.0)
    v = torch.randn((n, 3), generator=g, device="cuda", dtype=torch.float64)
    return (v * (r / torch.linalg.vector_norm(v, dim=1, keepdim=True))).float()


def prepare(case, seed):
    kind = case["kind"]
    if kind == "push":
        return _prepare_push(case, seed)
    if kind == "neural":
        spec, _, ctx, _ = _net_context(seed, _network(), 10.0)
        ctx.field_select(gcpush.FIELD_SIREN)
        ctx.inject([synth.EnsembleSpec(case["n"], lam_au=0.5, lat_deg=24.0, r_out_au=synth.r_out_default(spec))])
        return {"case": case, "ctx": ctx, "host": gcpush.state_buffers(ctx.n, alloc=_pinned)}
    if kind == "heldout":
        spec, nodes, ctx, _ = _net_context(seed, _network(), 10.0)
        n = case["n"]
        new = functools.partial(torch.empty, dtype=torch.float32, device="cuda")
        return {"case": case, "ctx": ctx, "x": _points(n, spec, seed), "t": new((n, 8)), "y": new((n, 8)),
                "J": new((n, 8, 3)), "spec": spec, "nodes": nodes}
    params = synth.siren_init(seed % 65521)
    spec, nodes, ctx, desc = _net_context(seed, params, synth.SIREN_OMEGA0, "main" if kind == "fit" else "small")
    s = {"case": case, "ctx": ctx, "x": _points(case["n"], spec, seed), "params": params, "desc": desc, "spec": spec,
         "nodes": nodes}
    if kind == "grad":
        s["t"] = torch.empty((case["n"], 8), dtype=torch.float32, device="cuda")
        ctx.field_targets(s["x"], s["t"])
        s["grad"] = torch.empty(N_SIREN, dtype=torch.float32, device="cuda")
    return s


# ------------------------------------------------------------------------------- one pass


def run(s):
    case, ctx = s["case"], s["ctx"]
    kind = case["kind"]
    if kind in ("push", "neural"):
        if case.get("restore"):
            ctx.set_state(s["host"])
        ctx.advance(0.5, case["steps"])
        out = {k: v.view(np.int32) if v.dtype == np.uint32 else v for k, v in ctx.get_state(out=s["host"]).items()}
        if case.get("tally"):
            out.update({k: v.view(np.int32 if v.dtype == np.uint32 else np.int64) for k, v in ctx.tally_read().items()})
        return out
    if kind == "heldout":
        ctx.field_targets(s["x"], s["t"])
        ctx.siren_eval(s["x"], s["y"], s["J"])
        return {"t": s["t"], "y": s["y"], "J": s["J"]}
    if kind == "grad":
        # the network is FP32 (BF16 products): its loss is a float32 number
        return {"loss": np.float32(ctx.siren_loss_grad(s["x"], s["t"], s["grad"])), "grad": s["grad"]}
    ctx.siren_set(s["params"], **s["desc"])
    loss = ctx.field_fit(s["x"], case["epochs"], batch=case["batch"], lr=1e-4)
    return {"loss": loss, "params": ctx.siren_get()}


def work(case):
    n, kind = case["n"], case["kind"]
    if kind in ("push", "neural"):
        if case.get("ens") == 64:
            n = synth.c3_batched().n_particles
        flop = 2 * 1_589_248 if kind == "neural" else 1019
        state = 172 * n
        if kind == "neural":
            return {"bytes": 2 * state + 404_000, "flops": n * case["steps"] * flop}
        wide = 2 if case["prec"] == "f64" else 1
        grid = 32 * wide * math.prod(GRIDS[case["grid"]]) * (2 if case["mode"] == "time" else 1)
        return {"bytes": 2 * state + min(grid, 16 * 32 * wide * n * case["steps"]), "flops": n * case["steps"] * flop}
    if kind == "heldout":
        return {"bytes": n * 4 * (3 + 8 + 8 + 24) + 404_000, "flops": n * 1_589_248}
    per_sample = 2 * (3 * 3 * 65536 + 3 * 2048 + 2 * 768)  # forward, weight and input gradients
    if kind == "grad":
        return {"bytes": n * 44 + 8 * N_SIREN, "flops": n * per_sample}
    rows = n // case["batch"] * case["batch"] * case["epochs"]
    return {"bytes": rows * 44 + 8 * N_SIREN, "flops": rows * per_sample}


# ------------------------------------------------------------------------------- 64 bits


def _layers(params):
    p = torch.as_tensor(params).cuda().double()
    w, b, o = [p[:768].view(256, 3)], [p[768:1024]], 1024
    for rows in (256, 256, 256, 8):
        w.append(p[o:o + 256 * rows].view(rows, 256))
        b.append(p[o + 256 * rows:o + 257 * rows])
        o += 257 * rows
    return w, b


def _net64(params, omega0, x):
    """Outputs and Jacobian of the network."""
    w, b = _layers(params)
    ys, js = [], []
    for q in x.double().split(65536):
        z = omega0 * (q @ w[0].T + b[0])
        h, d = torch.sin(z), (omega0 * torch.cos(z))[:, None, :] * w[0].T[None]
        for k in (1, 2, 3):
            z = h @ w[k].T + b[k]
            h, d = torch.sin(z), torch.cos(z)[:, None, :] * (d @ w[k].T)
        ys.append(h @ w[4].T + b[4])
        js.append((d @ w[4].T).transpose(1, 2))
    return torch.cat(ys), torch.cat(js)


def _grad64(params, omega0, x, t):
    """Mean squared error over samples and channels, and its gradient."""
    w, b = _layers(params)
    gw, gb, loss = [torch.zeros_like(v) for v in w], [torch.zeros_like(v) for v in b], 0.0
    for q, tt in zip(x.double().split(65536), t.double().split(65536)):
        zs, hs = [omega0 * (q @ w[0].T + b[0])], [q]
        for k in (1, 2, 3):
            hs.append(torch.sin(zs[-1]))
            zs.append(hs[-1] @ w[k].T + b[k])
        hs.append(torch.sin(zs[-1]))
        r = hs[4] @ w[4].T + b[4] - tt
        loss += float((r * r).sum()) / (8 * len(x))
        d = r / (4 * len(x))
        for k in (4, 3, 2, 1, 0):
            gw[k] += d.T @ hs[k]
            gb[k] += d.sum(0)
            if k:
                d = (d @ w[k]) * torch.cos(zs[k - 1]) * (omega0 if k == 1 else 1.0)
    return loss, torch.cat([v.reshape(-1) for pair in zip(gw, gb) for v in pair])


def _targets64(nodes, spec, x):
    """The grid's eight channels at x, interpolated and scaled as the network's outputs."""
    out = []
    for q in x.double().split(262144):
        pos = q * (spec.r_max_au * AU)
        rho, r = torch.hypot(pos[:, 0], pos[:, 1]), torch.linalg.vector_norm(pos, dim=1)
        fr = (r / AU - spec.r_min_au) / spec.dr_au
        ft = torch.atan2(rho, pos[:, 2]) * ((spec.n_th - 1) / math.pi)
        fp = torch.remainder(torch.atan2(pos[:, 1], pos[:, 0]), 2 * math.pi) * (spec.n_ph / (2 * math.pi))
        fr = fr.clamp(0, spec.n_r - 1)
        i, j, k = fr.floor().long().clamp(max=spec.n_r - 2), ft.floor().long().clamp(max=spec.n_th - 2), fp.floor().long()
        fr, ft, fp = fr - i, ft - j, fp - k
        v = 0.0
        for a in (0, 1):
            for b in (0, 1):
                for c in (0, 1):
                    wt = (fr if a else 1 - fr) * (ft if b else 1 - ft) * (fp if c else 1 - fp)
                    v = v + wt[:, None] * nodes[(k + c) % spec.n_ph, j + b, i + a].double()
        r = (r / AU)[:, None]
        out.append(torch.cat([v[:, :3] * r**2 / spec.B1, v[:, 3:6] * r / (spec.B1 * spec.u_sw),
                              v[:, 6:7] * r**2 / spec.B1, v[:, 7:] / (spec.B1 * spec.u_sw * AU)], 1))
    return torch.cat(out)


def exact(case, seed):
    """The network's and the interpolant's values in 64 bits. The pushes return none: a plain
    rendering of their many thousand dependent steps on the GPU takes over 20 seconds."""
    kind = case["kind"]
    if kind in ("push", "neural"):
        return None
    s = prepare(case, seed)
    if kind == "heldout":
        y, j = _net64(_network(), 10.0, s["x"])
        return {"t": _targets64(s["nodes"], s["spec"], s["x"]), "y": y, "J": j}
    w0 = s["desc"]["omega0"]
    if kind == "grad":
        loss, g = _grad64(s["params"], w0, s["x"], _targets64(s["nodes"], s["spec"], s["x"]))
        return {"loss": loss, "grad": g}
    t, b = _targets64(s["nodes"], s["spec"], s["x"]), case["batch"]
    p = torch.as_tensor(s["params"]).cuda().double()
    m, v, step, losses = torch.zeros_like(p), torch.zeros_like(p), 0, []
    for _ in range(case["epochs"]):
        mean = 0.0
        for k in range(case["n"] // b):
            loss, g = _grad64(p, w0, s["x"][k * b:k * b + b], t[k * b:k * b + b])
            step += 1
            m, v = 0.9 * m + 0.1 * g, 0.999 * v + 0.001 * g * g
            p = p - 1e-4 * (m / (1 - 0.9**step)) / (torch.sqrt(v / (1 - 0.999**step)) + 1e-8)
            mean += loss / (case["n"] // b)
        losses.append(mean)
    return {"loss": torch.tensor(losses, dtype=torch.float64), "params": p}
