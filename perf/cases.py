"""The work that users of this framework have it do, as measurable cases.

Every case goes through the package's public entry points: `solve` on one grid,
`solve_batched` and `Plan` on many, `eikonal` forward and backward, `eik_adjoint`,
`solve_slabs`, and the calls on host buffers.  All data are float64 (the only type the
solver has).  Inputs are made on the GPU from the seed alone: layered sections, smooth
random models, checkerboards and white noise, as in the benchmark and the tests.
"""
import math

import numpy as np
import torch

import paper_2103_05694_gb300 as eik

DEV = "cuda:0"


def listed():
    return [
        # one tiny 2D solve: launches and the latency of one short front
        {"name": "const_2d_129", "kind": "solve", "model": "const", "dims": "129x129", "h": 1.0 / 128.0, "nsrc": 1,
         "src_t": 0.0},
        # a small 3D block of strongly varying speeds, several sources with start times
        {"name": "noise_3d_small", "kind": "solve", "model": "noise", "dims": "20x21x22", "h": 0.5, "nsrc": 3,
         "src_t": 0.3},
        # one seismic section, one shot: a single long 2D front
        {"name": "layered_2d", "kind": "solve", "model": "layered", "dims": "751x2301", "h": 4.0, "nsrc": 1,
         "src_t": 0.0},
        # the same kind of section upsampled by 2 on each axis (nearest neighbour)
        {"name": "layered_2d_up2", "kind": "solve", "model": "layered2", "dims": "1502x4602", "h": 2.0, "nsrc": 1,
         "src_t": 0.0},
        # one large 3D volume with a 10:1 checkerboard
        {"name": "checker_3d_256", "kind": "solve", "model": "checker", "dims": "256x256x256", "h": 10.0, "nsrc": 1,
         "src_t": 0.0},
        # a 3D volume of odd, uneven sides, four sources with start times
        {"name": "smooth_3d_ragged", "kind": "solve", "model": "smooth", "dims": "97x131x203", "h": 10.0, "nsrc": 4,
         "src_t": 0.05},
        # 64 surface sources on one 128^3 model and 24 uneven grids: a plan replayed in a CUDA graph
        {"name": "batch_3d_graph", "kind": "plan", "model": "smooth", "side": 128, "lattice": 8, "grids": 24,
         "lo": 64, "hi": 192},
        # many uneven 2D sections in one call
        {"name": "batch_2d_ragged", "kind": "batch", "model": "smooth", "side": 0, "lattice": 0, "grids": 24,
         "lo": 65, "hi": 601},
        # one tomography step: 32 sources forward, misfit at the surface, gradient backward
        {"name": "tomography_2d_1024", "kind": "tomography", "n": 1024, "m": 1024, "nsrc": 32},
        # the adjoint alone, in 3D, with a dense misfit, gradients summed over the sources
        {"name": "adjoint_3d", "kind": "adjoint", "dims": "90x101x110", "nsrc": 8},
        # volumes in pinned host memory, solved into pinned host memory
        {"name": "host_3d_batch", "kind": "host", "model": "smooth", "side": 0, "lattice": 0, "grids": 4, "lo": 96,
         "hi": 160},
        # one section split into slabs with halo exchange
        {"name": "slabs_2d", "kind": "slabs", "model": "layered", "dims": "501x1201", "h": 4.0, "nsrc": 1, "slabs": 4},
    ]


def _log_int(rng, lo, hi):
    return min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi))))))


def draw(rng):
    kind = rng.choice(["solve2", "solve2", "solve3", "solve3", "plan", "batch", "tomography", "adjoint", "host",
                       "slabs"])
    if kind == "solve2":
        up = rng.random() < 0.3
        a, b = _log_int(rng, 24, 751), _log_int(rng, 32, 2301)
        model = rng.choice(["const", "noise", "smooth", "layered"])
        if up:
            return {"kind": "solve", "model": "layered2", "dims": "%dx%d" % (2 * a, 2 * b), "h": 2.0,
                    "nsrc": rng.choice([1, 1, 2]), "src_t": 0.0}
        return {"kind": "solve", "model": model, "dims": "%dx%d" % (a, b), "h": rng.choice([0.5, 4.0]),
                "nsrc": rng.choice([1, 1, 3, 12]), "src_t": rng.choice([0.0, 0.01])}
    if kind == "solve3":
        d = [_log_int(rng, 12, 240) for _ in range(3)]
        return {"kind": "solve", "model": rng.choice(["smooth", "checker", "noise"]), "dims": "%dx%dx%d" % tuple(d),
                "h": rng.choice([1.0, 10.0]), "nsrc": rng.choice([1, 2, 5, 16]), "src_t": rng.choice([0.0, 0.02])}
    if kind == "plan":
        return {"kind": "plan", "model": "smooth", "side": rng.randint(48, 112), "lattice": rng.randint(1, 8),
                "grids": rng.randint(0, 16), "lo": rng.randint(20, 60), "hi": rng.randint(80, 160)}
    if kind in ("batch", "host"):
        lattice, three_d = rng.randint(0, 3), kind == "host" or rng.random() < 0.3
        return {"kind": kind, "model": "smooth", "side": rng.randint(40, 120) if lattice and three_d else 0,
                "lattice": lattice if three_d else 0, "grids": rng.randint(2, 24 if kind == "batch" else 4),
                "lo": rng.randint(20, 90), "hi": rng.randint(100, 160 if three_d else 600)}
    if kind == "tomography":
        return {"kind": "tomography", "n": _log_int(rng, 64, 900), "m": _log_int(rng, 96, 1024),
                "nsrc": rng.choice([1, 3, 8, 20, 32])}
    if kind == "adjoint":
        two_d = rng.random() < 0.5
        d = [_log_int(rng, 40, 700) for _ in range(2)] if two_d else [_log_int(rng, 16, 110) for _ in range(3)]
        return {"kind": "adjoint", "dims": "x".join(str(x) for x in d), "nsrc": rng.randint(1, 9)}
    return {"kind": "slabs", "model": rng.choice(["layered", "smooth"]),
            "dims": "%dx%d" % (_log_int(rng, 40, 501), _log_int(rng, 60, 1201)), "h": 4.0, "nsrc": rng.choice([1, 3]),
            "slabs": rng.choice([2, 3, 4])}


# --- inputs -------------------------------------------------------------------------------------


def _dims(case):
    return tuple(int(x) for x in case["dims"].split("x"))


def _smooth_noise(gen, shape, sigma):
    """White noise under a Gaussian filter (periodic), mapped to [0, 1]."""
    f = torch.fft.rfftn(torch.randn(shape, generator=gen, device=DEV, dtype=torch.float64))
    for ax, n in enumerate(shape):
        k = torch.fft.rfftfreq(n, device=DEV, dtype=torch.float64) if ax == len(shape) - 1 else \
            torch.fft.fftfreq(n, device=DEV, dtype=torch.float64)
        w = torch.exp(-2.0 * (math.pi * sigma * k) ** 2)
        f = f * w.reshape([-1 if i == ax else 1 for i in range(len(shape))])
    g = torch.fft.irfftn(f, s=shape)
    return (g - g.min()) / (g.max() - g.min())


def _layered(gen, rng, nz, nx, h):
    """Sinusoidal layers from 1500 to 5500 m/s, three dipping faults, a smooth 5 % perturbation."""
    z = torch.arange(nz, device=DEV, dtype=torch.float64)[:, None] * h
    x = torch.arange(nx, device=DEV, dtype=torch.float64)[None, :] * h
    depth = z.expand(nz, nx)
    for _ in range(3):
        x0, dip, throw = rng.uniform(0, nx * h), math.radians(rng.uniform(55, 80)), rng.uniform(40, 200)
        depth = torch.where(x > x0 + z / math.tan(dip), depth - throw, depth)
    layer = torch.zeros((nz, nx), device=DEV, dtype=torch.int64)
    for k in range(12):
        base, amp = nz * h * (k + 1) / 13.0, rng.uniform(20, 80)
        lam, phase = rng.uniform(1000, 5000), rng.uniform(0, 2 * math.pi)
        layer += depth > base + amp * torch.sin(2 * math.pi * x / lam + phase)
    v = np.linspace(1500.0, 5500.0, 13) * (1.0 + rng.uniform(-0.05, 0.05, 13))
    v = torch.from_numpy(v).to(DEV)[layer]
    return (v * (1.0 + 0.2 * (_smooth_noise(gen, (nz, nx), 5.0) - 0.5))).clamp(1500.0, 5500.0)


def _speed(model, shape, h, gen, rng):
    if model == "const":
        return torch.full(shape, float(rng.uniform(1.0, 2.0)), device=DEV, dtype=torch.float64)
    if model == "noise":
        return 1.0 + 9.0 * torch.rand(shape, generator=gen, device=DEV, dtype=torch.float64)
    if model == "layered":
        return _layered(gen, rng, shape[0], shape[1], h)
    if model == "layered2":
        v = _layered(gen, rng, shape[0] // 2, shape[1] // 2, 2.0 * h)
        return v.repeat_interleave(2, 0).repeat_interleave(2, 1).contiguous()
    v = 1500.0 + 3000.0 * _smooth_noise(gen, shape, 8.0)
    if model == "checker":
        parity = torch.zeros(shape, device=DEV, dtype=torch.int64)
        inside = torch.ones(shape, device=DEV, dtype=torch.bool)
        for ax, n in enumerate(shape):
            i = torch.arange(n, device=DEV).reshape([-1 if a == ax else 1 for a in range(len(shape))])
            parity = parity + i // 16
            inside = inside & (i >= n // 4) & (i < n // 4 + n // 2)
        v = torch.where(inside & (parity % 2 == 1), v / 10.0, v)
    return v


def _rngs(seed):
    gen = torch.Generator(device=DEV)
    gen.manual_seed(int(seed))
    return gen, np.random.Generator(np.random.PCG64(int(seed)))


def _sources(model, shape, nsrc, src_t, rng):
    """Shots on the surface of sections and checkerboards, the middle of a constant grid, anywhere else."""
    n = int(np.prod(shape))
    if nsrc == 1 and model == "const":
        return [int(np.ravel_multi_index([s // 2 for s in shape], shape))], [0.0]
    plane = n // shape[0]
    if model in ("layered", "layered2") or (model == "checker" and nsrc == 1):
        idx = [int(i) for i in np.unique(rng.integers(plane // 4, max(plane // 4 + 1, 3 * plane // 4), nsrc))]
    else:
        idx = [int(i) for i in np.unique(rng.integers(0, n, nsrc))]
    return idx, [float(x) for x in rng.uniform(0.0, 1.0, len(idx)) * src_t]


def _grid(case, seed):
    gen, rng = _rngs(seed)
    shape = _dims(case)
    speed = _speed(case["model"], shape, case["h"], gen, rng)
    idx, t0 = _sources(case["model"], shape, case["nsrc"], case.get("src_t", 0.0), rng)
    return speed, idx, t0


def _uneven(case):
    """The shapes of the uneven grids of a batch: they go with the case, not with the seed."""
    lo, hi = case["lo"], case["hi"]
    rng = np.random.Generator(np.random.PCG64(1000 * hi + lo))
    if case["kind"] == "plan":
        return [(int(n),) * 3 for n in rng.integers(lo, hi + 1, case["grids"])]
    d = 3 if case["kind"] == "host" or case["lattice"] else 2
    return [tuple(int(n) for n in rng.integers(lo, hi + 1, d)) for _ in range(case["grids"])]


def _problems(case, seed):
    """(speed, sources) of a batch: one shared model under a lattice of surface sources, and uneven grids."""
    gen, rng = _rngs(seed)
    got = []
    if case["lattice"]:
        n, k = case["side"], case["lattice"]
        model = _speed("smooth", (n, n, n), 10.0, gen, rng)
        at = [(2 * i + 1) * n // (2 * k) for i in range(k)]
        got += [(model, [y * n + x]) for y in at for x in at]
    for shape in _uneven(case):
        idx = np.unique(rng.integers(0, int(np.prod(shape)), int(rng.integers(1, 5))))
        got.append((_speed("smooth", shape, 10.0, gen, rng), [int(i) for i in idx]))
    return got


def _tomography(case, seed):
    """Slowness, surface sources, receivers and observed times (straight rays, one per cent of noise)."""
    gen, rng = _rngs(seed)
    n, m, k = case["n"], case["m"], case["nsrc"]
    v = 2000.0 + 2000.0 * _smooth_noise(gen, (n, m), 16.0)
    src = [(2 * i + 1) * m // (2 * k) for i in range(k)]
    rcv = torch.arange(1, m, 2, device=DEV)
    dist = 5.0 * (rcv[None, :] - torch.tensor(src, device=DEV)[:, None]).abs().to(torch.float64)
    noise = torch.randn(dist.shape, generator=gen, device=DEV, dtype=torch.float64)
    return 1.0 / v, src, rcv, dist / 3000.0 * (1.0 + 0.01 * noise)


def _adjoint(case, seed):
    gen, rng = _rngs(seed)
    shape = _dims(case)
    speed = _speed("smooth", shape, 10.0, gen, rng)
    src = [[int(rng.integers(0, speed.numel()))] for _ in range(case["nsrc"])]
    g = torch.randn((len(src),) + shape, generator=gen, device=DEV, dtype=torch.float64)
    return speed, src, g


def _index(idx):
    return torch.tensor(idx, device=DEV, dtype=torch.int64)


def prepare(case, seed):
    kind = case["kind"]
    s = {"kind": kind}
    if kind in ("solve", "slabs"):
        speed, idx, t0 = _grid(case, seed)
        s.update(speed=speed, h=case["h"], src=_index(idx), out=torch.empty_like(speed))
        s["src_t"] = torch.tensor(t0, device=DEV, dtype=torch.float64) if any(t0) else None
        s["slabs"] = case.get("slabs", 0)
    elif kind in ("plan", "batch"):
        probs = _problems(case, seed)
        s["flat"] = torch.empty(sum(v.numel() for v, _ in probs), device=DEV, dtype=torch.float64)
        at, s["problems"] = 0, []
        for v, idx in probs:
            s["problems"].append({"speed": v, "h": 10.0, "sources": _index(idx),
                                  "out": s["flat"][at:at + v.numel()].view(v.shape)})
            at += v.numel()
        if kind == "plan":
            s["plan"] = eik.Plan(s["problems"])
            s["plan"].enqueue()
            s["plan"].status()
            s["graph"] = torch.cuda.CUDAGraph()
            with torch.cuda.graph(s["graph"]):
                s["plan"].enqueue()
    elif kind == "host":
        s["problems"] = [{"speed": v.cpu().pin_memory(), "h": 10.0, "sources": torch.tensor(idx, dtype=torch.int64),
                          "out": torch.empty(v.shape, dtype=torch.float64).pin_memory()}
                         for v, idx in _problems(case, seed)]
    elif kind == "tomography":
        slow, src, rcv, obs = _tomography(case, seed)
        s.update(slow=slow.requires_grad_(True), src=[_index([i]) for i in src], rcv=rcv, obs=obs)
    else:
        speed, src, g = _adjoint(case, seed)
        t = torch.empty_like(g)
        s["problems"] = [{"speed": speed, "h": 10.0, "sources": _index(i), "out": t[k]} for k, i in enumerate(src)]
        eik.solve_batched(s["problems"])
        s.update(g=[x for x in g], grad=torch.empty_like(speed))
    return s


def run(s):
    kind = s["kind"]
    if kind == "solve":
        return eik.solve(s["speed"], s["h"], s["src"], s["src_t"], out=s["out"]).t
    if kind == "slabs":
        return eik.solve_slabs(s["speed"], s["h"], s["src"], s["slabs"], out=s["out"]).t
    if kind == "plan":
        s["graph"].replay()
        return s["flat"]
    if kind == "batch":
        eik.solve_batched(s["problems"])
        return s["flat"]
    if kind == "host":
        eik.solve_batched(s["problems"])
        return [p["out"] for p in s["problems"]]
    if kind == "tomography":
        t = eik.eikonal(s["slow"], 5.0, s["src"])
        loss = 0.5 * ((t[:, 0, :][:, s["rcv"]] - s["obs"]) ** 2).sum()
        grad, = torch.autograd.grad(loss, s["slow"])
        return {"t": t.detach(), "loss": loss.detach(), "grad": grad}
    n = len(s["problems"])
    eik.eik_adjoint(s["problems"], s["g"], [s["grad"]] * n, {"sched_flags": eik.SUM_SHARED_GRADIENTS})
    return s["grad"]


# --- what a pass cannot do without ---------------------------------------------------------------


def work(case):
    kind = case["kind"]
    if kind in ("solve", "slabs"):
        shape = _dims(case)
        n = math.prod(shape)
        return {"bytes": 16 * n, "flops": n * (9 if len(shape) == 2 else 14)}
    if kind in ("plan", "batch", "host"):
        three_d = kind in ("plan", "host") or case["lattice"] > 0
        n, shared = sum(math.prod(x) for x in _uneven(case)), case["side"] ** 3 if case["lattice"] else 0
        cells = n + case["lattice"] ** 2 * shared
        return {"bytes": 8 * (n + shared) + 8 * cells, "flops": cells * (14 if three_d else 9)}
    if kind == "tomography":
        n, k = case["n"] * case["m"], case["nsrc"]
        return {"bytes": 8 * n * (2 + 3 * k), "flops": n * k * (9 + 10)}
    shape = _dims(case)
    n, k = math.prod(shape), case["nsrc"]
    return {"bytes": 8 * n * (2 + 2 * k), "flops": n * k * (10 if len(shape) == 2 else 14)}


# --- the same in plain torch ----------------------------------------------------------------------


def _minima(t, d):
    """The smaller neighbour on each of the last d axes (+inf off the grid)."""
    got = []
    for ax in range(t.dim() - d, t.dim()):
        p = torch.full_like(t, math.inf)
        n = t.shape[ax]
        if n > 1:
            p.narrow(ax, 1, n - 1).copy_(t.narrow(ax, 0, n - 1))
            q = p.narrow(ax, 0, n - 1)
            torch.minimum(q, t.narrow(ax, 1, n - 1), out=q)
        got.append(p)
    return got


def _fixed_point(r, sources, t0, d):
    """First-order upwind arrival times for r = h / v by plain iteration; leading axes are batches."""
    t = torch.full_like(r, math.inf)
    flat = t.view(len(sources), -1)
    fixed = torch.zeros_like(flat, dtype=torch.bool)
    for b, (idx, tt) in enumerate(zip(sources, t0)):
        for i, x in sorted(zip(idx, tt), key=lambda e: -e[1]):
            flat[b, i] = x
            fixed[b, i] = True
    fixed = fixed.view(t.shape)
    c = r * r
    while True:
        before = t.clone()
        for _ in range(32):
            a = _minima(t, d)
            lo, hi = torch.minimum(a[0], a[1]), torch.maximum(a[0], a[1])
            if d == 3:
                mid = torch.minimum(hi, a[2])
                top = torch.maximum(hi, a[2])
                lo, hi = torch.minimum(lo, mid), torch.maximum(lo, mid)
            b1 = hi - lo
            two = 0.5 * (b1 + (2.0 * c - b1 * b1).clamp_(min=0.0).sqrt_())
            u = torch.where(b1 < r, two, r)
            if d == 3:
                b2 = top - lo
                s, q = b1 + b2, b1 * b1 + b2 * b2
                three = (s + (s * s - 3.0 * (q - c)).clamp_(min=0.0).sqrt_()) / 3.0
                u = torch.where((b1 < r) & (b2 < two), three, u)
            t = torch.where(fixed, t, torch.minimum(t, lo + u))
        same = (before == t) | ((before - t) <= 1e-15 * t)
        if bool(same.all()):
            return t


def _gradient(r, h, t, g, sources, d):
    """Sum over the batch of d(loss)/d(slowness) by implicit differentiation of the local equations."""
    live = torch.isfinite(t)
    flat = live.view(len(sources), -1)
    for b, idx in enumerate(sources):
        flat[b, idx] = False
    a = _minima(t, d)
    m = [torch.where(live & (x < t), t - x, 0.0) for x in a]
    S = sum(m)
    S = torch.where(S > 0, S, math.inf)
    w = [x / S for x in m]
    lam = g.clone()
    axes = range(t.dim() - d, t.dim())
    share = []
    for k, ax in enumerate(axes):     # the weight each cell gives its lower and its upper neighbour
        n = t.shape[ax]
        lo, hi = torch.full_like(t, math.inf), torch.full_like(t, math.inf)
        lo.narrow(ax, 1, n - 1).copy_(t.narrow(ax, 0, n - 1))
        hi.narrow(ax, 0, n - 1).copy_(t.narrow(ax, 1, n - 1))
        half = torch.where(lo == hi, 0.5, 1.0)
        share.append((torch.where(lo == a[k], w[k] * half, 0.0), torch.where(hi == a[k], w[k] * half, 0.0)))
    while True:
        before = lam
        for _ in range(32):
            new = g.clone()
            for (lo, hi), ax in zip(share, axes):
                n = t.shape[ax]
                new.narrow(ax, 0, n - 1).add_((lam * lo).narrow(ax, 1, n - 1))
                new.narrow(ax, 1, n - 1).add_((lam * hi).narrow(ax, 0, n - 1))
            lam = new
        if bool(((lam - before).abs() <= 1e-15 * lam.abs()).all()):
            break
    return (torch.where(live, lam, 0.0) * (h * r) / S).sum(0)


def exact(case, seed):
    kind = case["kind"]
    if kind in ("solve", "slabs"):
        speed, idx, t0 = _grid(case, seed)
        if kind == "slabs":
            t0 = [0.0] * len(idx)
        return _fixed_point((case["h"] / speed)[None], [idx], [t0], speed.dim())[0]
    if kind in ("plan", "batch", "host"):
        probs, outs = _problems(case, seed), []
        k = case["lattice"] ** 2
        if k:
            v = probs[0][0]
            src = [p[1] for p in probs[:k]]
            r = (10.0 / v)[None].expand((k,) + tuple(v.shape)).contiguous()
            outs += list(_fixed_point(r, src, [[0.0]] * k, 3))
            del r
        for v, idx in probs[k:]:
            outs.append(_fixed_point((10.0 / v)[None], [idx], [[0.0] * len(idx)], v.dim())[0])
        return [x.cpu() for x in outs] if kind == "host" else torch.cat([x.reshape(-1) for x in outs])
    if kind == "tomography":
        slow, src, rcv, obs = _tomography(case, seed)
        src = [[i] for i in src]
        r = (5.0 * slow)[None].expand((len(src),) + tuple(slow.shape)).contiguous()
        t = _fixed_point(r, src, [[0.0]] * len(src), 2)
        miss = t[:, 0, :][:, rcv] - obs
        g = torch.zeros_like(t)
        g[:, 0, rcv] = miss
        return {"t": t, "loss": 0.5 * (miss ** 2).sum(), "grad": _gradient(r, 5.0, t, g, src, 2)}
    speed, src, g = _adjoint(case, seed)
    r = (10.0 / speed)[None].expand(g.shape).contiguous()
    t = _fixed_point(r, src, [[0.0]] * len(src), speed.dim())
    return _gradient(r, 10.0, t, g, src, speed.dim())
