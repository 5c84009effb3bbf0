"""Performance cases of the library: what a program does with it, through its public entry points.

The kinds of work:

* ``step``     forward simulation: set_state, ``Scene.step(n)``, get_state
* ``rollout``  a differentiable rollout with its reverse pass through ``rollout.rollout`` (the
               torch.autograd function), checkpointed every ``ckpt`` steps (1: every state kept)
* ``material`` system identification: per-particle stiffness and mass, slip walls with friction,
               ``Scene.rollout`` / ``Scene.backward`` and the material gradients
* ``batch``    a serving batch: many small requests of uneven size and horizon, some with their
               gradient, advanced together (``Batch``)
* ``noalloc``  a control loop on the allocation-free step ``mpm_step_noalloc``
* ``fp64``     an accuracy study in double precision (``Scene64``): host arrays in and out

Scenes are unions of random boxes on the floor of the grid (two discs for ``fp64``), seeded on a
jittered lattice, in motion and slightly deformed.  ``exact`` is the same step in float64 torch,
differentiated by autograd.
"""
import ctypes
import math

import numpy as np
import torch

from paper_1810_01054_gb300 import mpm, rollout, scenes

# Sizes follow the repository's workloads: the 1,024-particle square, the 2D walker (31,458
# particles, 16 per cell), the 3D soft body (95,123 particles, MLP controller), the 3D cluster (one
# million particles, 64 groups), the serving mix, the colliding discs.
_LISTED = [
    # smallest: an interactive 2D scene, a few particles per cell, launches and latency only
    dict(name="step_square2d", kind="step", dim=2, nx=64, ny=64, nz=1, particles=1024, per_axis=2, steps=64,
         ckpt=0, ctrl="sin", groups=2, hidden=0, walls="sticky"),
    # its gradient: trajectory optimisation of a small body, every state kept
    dict(name="grad_square2d", kind="rollout", dim=2, nx=64, ny=64, nz=1, particles=1024, per_axis=2, steps=48,
         ckpt=1, ctrl="table", groups=2, hidden=48, walls="sticky"),
    # the 2D walker, simulated
    dict(name="step_walker2d", kind="step", dim=2, nx=128, ny=128, nz=1, particles=31458, per_axis=4, steps=48,
         ckpt=0, ctrl="basis", groups=4, hidden=0, walls="sticky"),
    # the 2D walker, one training rollout of its controller with checkpoints
    dict(name="grad_walker2d", kind="rollout", dim=2, nx=128, ny=128, nz=1, particles=31458, per_axis=4, steps=48,
         ckpt=16, ctrl="basis", groups=4, hidden=0, walls="sticky"),
    # odd sizes: a small 3D body on a grid whose sides are no multiples of anything, closed-loop controller
    dict(name="grad_ragged3d", kind="rollout", dim=3, nx=37, ny=53, nz=41, particles=7919, per_axis=2, steps=24,
         ckpt=1, ctrl="com", groups=5, hidden=0, walls="slip"),
    # the 3D soft body: training its MLP controller with checkpoints
    dict(name="grad_soft3d", kind="rollout", dim=3, nx=64, ny=64, nz=64, particles=95123, per_axis=2, steps=24,
         ckpt=5, ctrl="mlp", groups=16, hidden=64, walls="sticky"),
    # inference of material parameters on a mid-sized 3D body
    dict(name="material3d", kind="material", dim=3, nx=64, ny=64, nz=64, particles=64000, per_axis=2, steps=16,
         ckpt=4, ctrl="sin", groups=1, hidden=0, walls="slip"),
    # the large 3D scene, simulated
    dict(name="step_cluster3d", kind="step", dim=3, nx=128, ny=128, nz=128, particles=1000000, per_axis=2, steps=16,
         ckpt=0, ctrl="sin", groups=64, hidden=0, walls="sticky"),
    # the large 3D scene, its gradient with checkpoints
    dict(name="grad_cluster3d", kind="rollout", dim=3, nx=128, ny=128, nz=128, particles=1000000, per_axis=2,
         steps=12, ckpt=4, ctrl="sin", groups=64, hidden=0, walls="sticky"),
    # serving: small 2D requests of uneven size and horizon in one batch
    dict(name="batch_mix2d", kind="batch", dim=2, nx=64, ny=64, nz=1, particles=24000, per_axis=2, steps=40,
         ckpt=0, ctrl="sin", groups=16, hidden=0, walls="sticky", requests=16),
    # a control loop that must not allocate: one step per call
    dict(name="noalloc_loop3d", kind="noalloc", dim=3, nx=64, ny=64, nz=64, particles=95123, per_axis=2, steps=8,
         ckpt=0, ctrl="table", groups=16, hidden=8, walls="sticky"),
    # the accuracy study: two colliding discs in double precision, every step's actuation a variable
    dict(name="fp64_discs2d", kind="fp64", dim=2, nx=64, ny=64, nz=1, particles=628, per_axis=2, steps=50,
         ckpt=0, ctrl="table", groups=2, hidden=50, walls="sticky"),
]


def listed():
    return [dict(c) for c in _LISTED]


def _log_uniform(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["step", "step", "step", "rollout", "rollout", "rollout", "material", "batch", "noalloc", "fp64"])
    dim = 2 if kind in ("batch", "fp64") else rng.choice([2, 3, 3])
    per_axis = 2 if dim == 3 or kind in ("batch", "fp64") else rng.choice([2, 4])
    hi = 15000 * per_axis - 15000 if dim == 2 else 1000000
    hi = {"batch": 60000, "fp64": 1500}.get(kind, min(hi, {"noalloc": 150000, "material": 250000}.get(kind, hi)))
    lo = {"batch": 6000, "fp64": 300}.get(kind, 700 if dim == 2 else 2000)
    particles = _log_uniform(rng, lo, hi)
    # a grid that the body fills to between a twentieth and a quarter (a batch: each of its requests)
    requests = rng.randint(8, 24) if kind == "batch" else 0
    cells = particles / float(max(1, requests)) / per_axis ** dim
    side = (cells / math.exp(rng.uniform(math.log(0.05), math.log(0.25)))) ** (1.0 / dim)
    if kind == "fp64":
        sides = [64, 64, 1]
    else:
        top = 63 if kind == "noalloc" and dim == 3 else 128
        sides = [min(top, max(28, int(side * rng.uniform(0.85, 1.2)) + 10)) for _ in range(dim)] + [1] * (3 - dim)
    ctrl = "table" if kind in ("noalloc", "fp64") else "sin" if kind in ("batch", "material") else rng.choice(
        ["sin", "basis", "mlp", "table", "com"])
    groups = 2 if kind == "fp64" else rng.choice([1, 3, 4, 16] if ctrl in ("mlp", "com") else [1, 2, 4, 16, 64])
    # a pass of no more particle-steps (with their reverse steps) than the largest listed case
    weight = 4 if kind in ("rollout", "material", "batch") else 1.5
    most = max(8, min(48, int(40e6 / (weight * particles))))
    steps = rng.randint(8, most)
    ckpt = 0 if kind not in ("rollout", "material") else rng.choice([1, 1, 4, 7])
    return dict(kind=kind, dim=dim, nx=sides[0], ny=sides[1], nz=sides[2], particles=particles, per_axis=per_axis,
                steps=steps, ckpt=ckpt, ctrl=ctrl, groups=groups,
                hidden={"table": steps, "mlp": rng.choice([16, 64])}.get(ctrl, 0),
                walls=rng.choice(["sticky", "slip"]) if kind not in ("batch", "fp64") else "sticky", requests=requests)


# ------------------------------------------------------------------------------------- scenes
_DEV = "cuda"
_ctx = None


def _context():
    """One context on torch's current stream, as a program with torch tensors keeps it."""
    global _ctx
    if _ctx is None:
        _ctx = mpm.Context(0, stream=torch.cuda.current_stream())
    return _ctx


def _grid(case):
    return tuple(int(case[k]) for k in ("nx", "ny", "nz"))[: case["dim"]]


def _generator(*seed):
    g = torch.Generator(device=_DEV)
    g.manual_seed(int(np.random.SeedSequence([int(s) for s in seed]).generate_state(1, np.uint64)[0] >> 1))
    return g


def _rand(g, *shape):
    return torch.rand(*shape, generator=g, device=_DEV, dtype=torch.float64)


def _boxes(g, grid, dx, per_axis, count):
    """`count` lattice points (spacing dx / per_axis) of a union of random boxes on the floor."""
    dim = len(grid)
    first = [3] * dim  # the floor: three cells above the grid's end; the same margin elsewhere
    size = [(n - 8) * per_axis for n in grid]
    taken = torch.zeros(size, dtype=torch.bool, device=_DEV)
    parts, have = [], 0
    for _ in range(300):
        if have >= count:
            break
        r = _rand(g, 2, dim).cpu().numpy()
        ext = [max(per_axis, int(size[a] * (0.2 + 0.3 * r[0, a]))) for a in range(dim)]
        lo = [0 if a == 1 else int((size[a] - ext[a]) * r[1, a]) for a in range(dim)]
        box = tuple(slice(lo[a], lo[a] + ext[a]) for a in range(dim))
        fresh = (~taken[box]).nonzero()[: count - have]
        taken[box] = True
        parts.append(fresh + torch.tensor(lo, device=_DEV))
        have += fresh.shape[0]
    if have < count:  # the boxes cover one another: the lowest free points
        free = (~taken).transpose(0, 1).nonzero()[: count - have]
        parts.append(free[:, [1, 0, 2][:dim]])
        have += free.shape[0]
    if have < count:
        raise ValueError("the grid has no room for %d particles" % count)
    s = dx / per_axis
    pts = torch.cat(parts).double()
    corner = torch.tensor([f * dx for f in first], device=_DEV, dtype=torch.float64)
    return corner + (pts + 0.5 + 0.2 * (_rand(g, *pts.shape) - 0.5)) * s


def _discs(g, dx, count):
    """About to collide: `count` points of two discs of one size, the left one first."""
    half = [count - count // 2, count // 2]
    R = dx * math.sqrt(half[0] / 4.0 / math.pi)
    s, out = dx / 2, []
    for k, c in enumerate((torch.tensor([0.35, 0.45]), torch.tensor([0.35 + 2 * R + 1.0 * dx, 0.45 + 0.35 * R]))):
        r = int(R / s) + 3
        ii = torch.arange(-r, r + 1, dtype=torch.float64)
        p = torch.stack(torch.meshgrid(ii, ii, indexing="ij"), -1).reshape(-1, 2) + 0.25
        p = p[p.norm(dim=1).argsort(stable=True)[: half[k]]]
        out.append(c.double() + p * s)
    pts = torch.cat(out).to(_DEV)
    return pts + 0.2 * (_rand(g, *pts.shape) - 0.5) * s


def _waves(g, x, rows, amplitude, modes=(1.0, 2.0)):
    """`rows` smooth fields of x, each a sum of two waves, and their gradients [N, rows, dim]."""
    dim = x.shape[1]
    val = torch.zeros(x.shape[0], rows, device=_DEV, dtype=torch.float64)
    grad = torch.zeros(x.shape[0], rows, dim, device=_DEV, dtype=torch.float64)
    for m in modes:
        k = 2 * math.pi * m * (2 * _rand(g, rows, dim) - 1)
        ph = 2 * math.pi * _rand(g, rows)
        u = x @ k.T + ph
        a = amplitude / (2 * m)
        val += a * u.sin()
        grad += (a * u.cos())[:, :, None] * k
    return val, grad


def _inputs(case, seed, particles=None, grid=None):
    """Everything a scene is made of, as float32-valued float64 tensors and plain numbers."""
    dim, per = case["dim"], case["per_axis"]
    grid = grid or _grid(case)
    N = particles or case["particles"]
    g = _generator(seed, dim, N, *grid)
    f32 = lambda t: t.float().double()  # noqa: E731
    dx = 1.0 / (64 if max(grid) <= 64 else 128)
    discs = case["kind"] == "fp64"
    E = 100.0 if discs else 20.0 if dim == 2 else 50.0
    dt = 2e-4 if dim == 3 and max(grid) > 64 else 5e-4
    x = f32(_discs(g, dx, N) if discs else _boxes(g, grid, dx, per, N))
    d2 = dim * dim
    if discs:
        v = torch.zeros_like(x)
        v[: N - N // 2, 0] = 0.6
        C = torch.zeros(N, dim, dim, device=_DEV, dtype=torch.float64)
        v = v + _waves(g, x, dim, 0.02)[0]
    else:
        v, C = _waves(g, x, dim, 2.0, (2.0, 4.0))
    F = torch.eye(dim, device=_DEV, dtype=torch.float64) + _waves(g, x, d2, 0.08)[0].reshape(N, dim, dim)
    if case["groups"] > 0:
        if discs:
            group = (torch.arange(N, device=_DEV) >= N - N // 2).int()
        else:  # slices of the body along its first axis
            q = (x[:, 0] - x[:, 0].min()) / (x[:, 0].max() - x[:, 0].min() + 1e-12)
            group = (q * case["groups"]).int().clamp_(max=case["groups"] - 1)
            group[x[:, 1] > x[:, 1].quantile(0.8) if N <= 1 << 24 else x[:, 1] > 1] = -1
    else:
        group = torch.full((N,), -1, dtype=torch.int32, device=_DEV)
    G, H = case["groups"], case["hidden"]
    rng = np.random.default_rng([int(seed), dim, N, 7])
    ctrl = {"sin": scenes.CTRL_SIN, "basis": scenes.CTRL_BASIS, "mlp": scenes.CTRL_MLP, "table": scenes.CTRL_TABLE,
            "com": scenes.CTRL_COM}[case["ctrl"]]
    amp, scale = E / 8, 1.0
    if case["ctrl"] == "mlp":
        params, scale = scenes.mlp_init(rng, G, dim, H), E / 4
    elif case["ctrl"] == "com":
        params, scale = scenes.com_init(rng, G, dim, [0.6] * dim), E / 4
    else:
        params = amp * rng.uniform(-1, 1, scenes.n_ctrl_params(ctrl, G, dim, H))
    dirs = np.zeros((G, dim))
    dirs[:, 1] = 1.0
    vol = float(np.float32((dx / per) ** dim))
    spec = dict(dim=dim, grid=grid, dx=float(np.float32(dx)), dt=float(np.float32(dt)), E=E, nu=float(np.float32(0.3)),
                vol=vol, mass=vol, gravity=[0.0 if discs or a != 1 else float(np.float32(-9.8)) for a in range(dim)],
                kind=[0] * (2 * dim), c=[0.0] * (2 * dim), width=3, x=x, v=f32(v), C=f32(C), F=f32(F), group=group,
                dirs=dirs, ctrl=case["ctrl"], ctrl_id=ctrl, G=G, H=H, freq=2.0, scale=scale,
                params=f32(torch.tensor(params, device=_DEV)), Ep=None, mp=None)
    if case["walls"] == "slip":  # a sticky floor, slip walls of different friction around it
        spec["kind"] = [0 if w == 2 else 1 for w in range(2 * dim)]
        spec["c"] = [0.0 if w == 2 else float(np.float32(0.1 + 0.1 * w)) for w in range(2 * dim)]
    if case["kind"] == "material":
        spec["Ep"] = f32(E * (0.8 + 0.4 * _rand(g, N)))
        spec["mp"] = f32(vol * (0.8 + 0.4 * _rand(g, N)))
    # dL/d(final state): a tracking loss on positions and velocities, different for every particle
    s = _waves(g, x, 2 * dim, 1.0)[0] + 0.5 * (2 * _rand(g, N, 2 * dim) - 1)
    spec["gx"], spec["gv"] = f32(s[:, :dim] / N), f32(0.05 * s[:, dim:] / N)
    return spec


def _scene_spec(p, name, fp64=False):
    """The library's scene description of these inputs (device arrays; host arrays for FP64)."""
    conv = (lambda t: t.cpu().numpy()) if fp64 else (lambda t: t.float())
    slip = any(p["kind"])
    return scenes.SceneSpec(
        name=name, dim=p["dim"], n_grid=p["grid"], dx=p["dx"], dt=p["dt"], gravity=tuple(p["gravity"]), E=p["E"],
        nu=p["nu"], p_mass=p["mass"], p_vol=p["vol"], bc_type=scenes.BC_STICKY, bc_width=p["width"], friction_c=0.0,
        x0=conv(p["x"]), v0=conv(p["v"]), C0=conv(p["C"]), F0=conv(p["F"]),
        group=p["group"].cpu().numpy() if fp64 else p["group"], act_dir=p["dirs"], ctrl_type=p["ctrl_id"],
        ctrl_params=p["params"].cpu().numpy(), ctrl_hidden=p["H"], ctrl_freq=p["freq"], ctrl_scale=p["scale"],
        E_arr=None if p["Ep"] is None else p["Ep"].float(), mass_arr=None if p["mp"] is None else p["mp"].float(),
        wall_kind=np.array(p["kind"], np.int32) if slip else None,
        wall_c=np.array(p["c"], np.float32) if slip else None)


def _state_buffers(N, dim):
    e = lambda *s: torch.empty(s, device=_DEV)  # noqa: E731
    return e(N, dim), e(N, dim), e(N, dim, dim), e(N, dim, dim)


def _batch_requests(case):
    """Sizes and horizons of the batch's requests: shares of the total, two in three with gradient."""
    rng = np.random.default_rng([case["particles"], 11])
    n, total = case["requests"], case["particles"]
    share = np.exp(rng.uniform(0.0, math.log(6.0), n))
    got = []
    for i in range(n):
        N = max(64, int(total * share[i] / share.sum()))
        T = int(case["steps"] * rng.uniform(0.5, 1.0)) + 1
        got.append((i, N, T, i % 3 != 2))
    return got


# ------------------------------------------------------------------------------------- prepare, run
def prepare(case, seed):
    kind, dim, N = case["kind"], case["dim"], case["particles"]
    ctx = _context()
    state = dict(case=case)
    if kind == "batch":
        state["requests"] = []
        for i, n, T, grad in _batch_requests(case):
            p = _inputs(case, seed * 1000 + i, particles=n)
            sc = mpm.Scene(ctx, _scene_spec(p, "request_%d" % i))
            start = [p[k].float() for k in ("x", "v", "C", "F")]
            out = _state_buffers(n, dim)
            gout = _state_buffers(n, dim) + (torch.empty(max(1, sc.n_params), device=_DEV),) if grad else None
            state["requests"].append((sc, T, grad, start, out, gout))
        edges = sorted({sc.tile_edge for sc, *_ in state["requests"]})
        state["batches"] = {e: mpm.Batch(ctx, dim) for e in edges}  # a batch per tile edge, as the server keeps them
        return state
    p = _inputs(case, seed)
    if kind == "fp64":
        spec = _scene_spec(p, "discs", fp64=True)
        state.update(scene=mpm.Scene64(ctx, spec), gx=p["gx"].cpu().numpy(), gv=p["gv"].cpu().numpy(),
                     x=spec.x0, v=spec.v0, F=spec.F0)
        return state
    start = [p[k].float() for k in ("x", "v", "C", "F")]
    if kind == "noalloc":
        bufs = [_state_buffers(N, dim), _state_buffers(N, dim)]
        acts = p["params"].float().reshape(case["hidden"], case["groups"]).contiguous()
        dirs = torch.tensor(p["dirs"], device=_DEV, dtype=torch.float32)
        status = torch.zeros(1, dtype=torch.int32, device=_DEV)
        calls = []
        for n in range(case["steps"]):
            src, dst = start if n == 0 else bufs[(n - 1) & 1], bufs[n & 1]
            a = mpm.NoAllocStep()
            a.device, a.dim, a.n_particles, a.n_groups = -1, dim, N, case["groups"]
            for k in range(3):
                a.n_grid[k] = p["grid"][k] if k < dim else 1
                a.gravity[k] = p["gravity"][k] if k < dim else 0.0
            a.dx, a.dt, a.E, a.nu, a.p_mass, a.p_vol = p["dx"], p["dt"], p["E"], p["nu"], p["mass"], p["vol"]
            a.bc_type, a.bc_width, a.friction_c = (1, 3, 0.2) if case["walls"] == "slip" else (0, 3, 0.0)
            a.x, a.v, a.C, a.F = (t.data_ptr() for t in src)
            a.x_out, a.v_out, a.C_out, a.F_out = (t.data_ptr() for t in dst)
            a.group, a.act_dir, a.act = p["group"].data_ptr(), dirs.data_ptr(), acts[n % len(acts)].data_ptr()
            a.status = status.data_ptr()
            calls.append(a)
        state.update(calls=calls, out=bufs[(case["steps"] - 1) & 1], keep=(start, bufs, acts, dirs, status, p["group"]),
                     stream=ctypes.c_void_p(torch.cuda.current_stream().cuda_stream))
        return state
    sc = mpm.Scene(ctx, _scene_spec(p, kind))
    state.update(scene=sc, start=start)
    if kind == "step":
        state["out"] = _state_buffers(N, dim)
    elif kind == "rollout":
        state["leaves"] = [t.clone().requires_grad_(True) for t in start + [p["params"].float()]]
        state["seeds"] = [p["gx"].float(), p["gv"].float(), torch.zeros(N, dim, dim, device=_DEV),
                          torch.zeros(N, dim, dim, device=_DEV)]
    else:
        state.update(out=_state_buffers(N, dim), gx=p["gx"].float(), gv=p["gv"].float(),
                     gout=_state_buffers(N, dim) + (torch.empty(max(1, sc.n_params), device=_DEV),))
    return state


def run(state):
    case = state["case"]
    kind, T = case["kind"], case["steps"]
    if kind == "step":
        sc = state["scene"]
        sc.set_state(*state["start"], step=0)
        sc.step(T)
        return list(sc.get_state(out=state["out"]))
    if kind == "rollout":
        leaves = state["leaves"]
        final = rollout.rollout(state["scene"], T, *leaves, ckpt_interval=case["ckpt"])
        grads = torch.autograd.grad(final, leaves, grad_outputs=state["seeds"])
        return [t.detach() for t in final] + list(grads)
    if kind == "material":
        sc = state["scene"]
        sc.set_state(*state["start"], step=0)
        sc.rollout(T, case["ckpt"])
        out = list(sc.get_state(out=state["out"]))
        grads = list(sc.backward(gx=state["gx"], gv=state["gv"], out=state["gout"]))
        return out + grads + list(sc.material_gradients())
    if kind == "batch":
        open_ = []
        for sc, steps, grad, start, out, gout in state["requests"]:
            sc.set_state(*start, step=0)
            b = state["batches"][sc.tile_edge]
            open_.append((b, b.admit(sc, steps, grad), sc, grad, out, gout))
        done = []
        waiting = list(open_)
        while waiting:
            for b in state["batches"].values():
                b.tick(8)
            still = []
            for w in waiting:
                (done if w[0].poll(w[1]) else still).append(w)
            waiting = still
        for b, slot, *_ in done:
            b.release(slot)
        answers = []
        for _, _, sc, grad, out, gout in open_:
            answers += list(sc.get_state(out=out))
            if grad:
                answers += list(sc.gradients(out=gout))
        return _by_kind(answers, open_)
    if kind == "noalloc":
        lib, stream = mpm.lib(), state["stream"]
        for a in state["calls"]:
            rc = lib.mpm_step_noalloc(ctypes.byref(a), stream)
            if rc != mpm.MPM_OK:
                raise mpm.MPMError(rc, "mpm_step_noalloc")
        return list(state["out"])
    sc = state["scene"]  # fp64
    sc.set_state(state["x"], state["v"], None, state["F"])
    sc.rollout(T)
    return list(sc.get_state()) + list(sc.backward(gx=state["gx"], gv=state["gv"]))


def _by_kind(answers, requests):
    """The requests' answers, all of one kind in one tensor: x, v, C, F, dL/d(x, v, C, F, params)."""
    parts = [[] for _ in range(9)]
    i = 0
    for _, _, _, grad, _, _ in requests:
        for k in range(9 if grad else 4):
            parts[k].append(answers[i].reshape(-1))
            i += 1
    return [torch.cat(q) for q in parts]


def work(case):
    """Per forward step the state read and written; per reverse step the state, the adjoint in and
    the adjoint out (a checkpointed rollout's recompute is no work of its own)."""
    dim, N, T = case["dim"], case["particles"], case["steps"]
    size = 8 if case["kind"] == "fp64" else 4
    S = 2 * dim + 2 * dim * dim
    nodes = 3 ** dim
    fwd_b, rev_b = 2 * S * size, 3 * S * size
    # forward: affine scatter and gather per node, stress and updates; reverse: about three times that
    fwd_f = nodes * (4 * dim * dim + 8 * dim + 4) + 30 * dim * dim
    rev_f = 3 * fwd_f
    if case["kind"] == "batch":
        T = 0.77 * T
        return {"bytes": N * T * (fwd_b + rev_b * 2 / 3), "flops": N * T * (fwd_f + rev_f * 2 / 3)}
    grad = case["kind"] in ("rollout", "material", "fp64")
    return {"bytes": float(N * T * (fwd_b + (rev_b if grad else 0))),
            "flops": float(N * T * (fwd_f + (rev_f if grad else 0)))}


# ------------------------------------------------------------------------------------- float64
def _cofactor(F):
    if F.shape[-1] == 2:
        rows = [torch.stack([F[:, 1, 1], -F[:, 1, 0]], -1), torch.stack([-F[:, 0, 1], F[:, 0, 0]], -1)]
    else:
        rows = [torch.linalg.cross(F[:, (i + 1) % 3], F[:, (i + 2) % 3]) for i in range(3)]
    return torch.stack(rows, 1)


def _walls64(p, v):
    """Boundary of the node velocities v [nodes, dim]: sticky bands, else the slip projections."""
    dim, grid = p["dim"], p["grid"]
    idx = torch.stack(torch.meshgrid(*[torch.arange(n, device=_DEV) for n in grid], indexing="ij"), -1).reshape(-1, dim)
    hit = [(idx[:, w // 2] >= grid[w // 2] - p["width"]) if w & 1 else (idx[:, w // 2] < p["width"])
           for w in range(2 * dim)]
    fixed = torch.zeros(v.shape[0], dtype=torch.bool, device=_DEV)
    for w in range(2 * dim):
        if p["kind"][w] == 0:
            fixed = fixed | hit[w]
    for w in range(2 * dim):
        if p["kind"][w] != 1:
            continue
        sgn = -1.0 if w & 1 else 1.0
        n = torch.zeros(dim, device=_DEV, dtype=torch.float64)
        n[w // 2] = sgn
        ln = v[:, w // 2] * sgn
        vt = v - ln[:, None] * n
        lt = (vt.square().sum(1) + 1e-20).sqrt()
        scale = (lt + p["c"][w] * ln.clamp(max=0)).clamp(min=0) / lt
        slid = scale[:, None] * vt + ln.clamp(min=0)[:, None] * n
        v = torch.where((hit[w] & ~fixed)[:, None], slid, v)
    return torch.where(fixed[:, None], torch.zeros_like(v), v)


def _actuation64(p, n, x, v, params):
    G, dim, t = p["G"], p["dim"], n * p["dt"]
    if G == 0:
        return None
    w = 2 * math.pi * p["freq"] * t
    if p["ctrl"] == "sin":
        return params * math.sin(w)
    if p["ctrl"] == "basis":
        b = torch.tensor([math.sin(w), math.cos(w), math.sin(2 * w), math.cos(2 * w)], device=_DEV, dtype=torch.float64)
        return params.reshape(G, 4) @ b
    if p["ctrl"] == "table":
        return params.reshape(-1, G)[n] if n < p["H"] else torch.zeros(G, device=_DEV, dtype=torch.float64)
    on = (p["group"][None, :] == torch.arange(G, device=_DEV)[:, None]).double()
    on = on / on.sum(1, keepdim=True).clamp(min=1)
    if p["ctrl"] == "com":
        Z = dim * (1 + 2 * G)
        z = torch.cat([params[:dim], (on @ x).reshape(-1), (on @ v).reshape(-1)])
        return p["scale"] * torch.tanh(params[dim: dim + G * Z].reshape(G, Z) @ z + params[dim + G * Z:])
    H, Z, o = p["H"], G * dim, 0
    empty = (p["group"][None, :] == torch.arange(G, device=_DEV)[:, None]).sum(1) == 0
    c = torch.where(empty[:, None], torch.zeros((), device=_DEV, dtype=torch.float64), on @ x)
    h = (c - x.mean(0)).reshape(-1)
    for rows, cols in ((H, Z), (H, H), (G, H)):
        W, b = params[o: o + rows * cols].reshape(rows, cols), params[o + rows * cols: o + rows * cols + rows]
        o += rows * cols + rows
        h = torch.tanh(W @ h + b)
    return p["scale"] * h


def _step64(p, n, x, v, C, F, params, Ep, mp):
    """One step of the method in float64, differentiable."""
    dim, grid, dx, dt = p["dim"], p["grid"], p["dx"], p["dt"]
    E = p["E"] if Ep is None else Ep[:, None, None]
    m = torch.full((x.shape[0], 1), p["mass"], device=_DEV, dtype=torch.float64) if mp is None else mp[:, None]
    mu, la = E / (2 * (1 + p["nu"])), E * p["nu"] / ((1 + p["nu"]) * (1 - 2 * p["nu"]))
    cof = _cofactor(F)
    J = (F[:, 0] * cof[:, 0]).sum(1)[:, None, None]
    Fit = cof / J
    P = mu * (F - Fit) + la * J.log() * Fit
    act = _actuation64(p, n, x, v, params)
    if act is not None:
        a = torch.cat([act, act.new_zeros(1)])[p["group"].long()]  # group -1: the zero at the end
        d = torch.cat([torch.tensor(p["dirs"], device=_DEV), act.new_zeros(1, dim)])[p["group"].long()]
        P = P + F * (a[:, None] * d)[:, None, :]
    Gm = -4.0 / dx ** 2 * dt * p["vol"] * P @ F.transpose(1, 2) + m[:, :, None] * C
    base = (x.detach() / dx - 0.5).floor()
    f = x / dx - base
    w = [0.5 * (1.5 - f).square(), 0.75 - (f - 1).square(), 0.5 * (f - 0.5).square()]
    lin = torch.zeros(x.shape[0], dtype=torch.long, device=_DEV)
    for a in range(dim):
        lin = lin * grid[a] + base[:, a].long()
    nodes = []
    for k in np.ndindex(*(3,) * dim):
        shift = 0
        N = torch.ones_like(m)
        for a in range(dim):
            shift = shift * grid[a] + k[a]
            N = N * w[k[a]][:, a: a + 1]
        nodes.append((lin + shift, N, (torch.tensor(k, device=_DEV, dtype=torch.float64) - f) * dx))
    field = torch.zeros(int(np.prod(grid)), dim + 1, device=_DEV, dtype=torch.float64)
    for i, N, d in nodes:
        mom = m * v + (Gm @ d[:, :, None])[:, :, 0]
        field = field.index_add(0, i, N * torch.cat([mom, m], 1))
    mass = field[:, dim:]
    live = mass > 0
    g = torch.tensor(p["gravity"], device=_DEV, dtype=torch.float64)
    vi = field[:, :dim] / torch.where(live, mass, torch.ones_like(mass)) + dt * g
    vi = torch.where(live, _walls64(p, vi), torch.zeros_like(vi))
    vn, Cn = torch.zeros_like(v), torch.zeros_like(C)
    for i, N, d in nodes:
        u = N * vi[i]
        vn = vn + u
        Cn = Cn + u[:, :, None] * d[:, None, :]
    Cn = 4.0 / dx ** 2 * Cn
    return x + dt * vn, vn, Cn, F + dt * Cn @ F


def _reference(p, T, grad, mean_seed=False):
    """x, v, C, F after T steps and, with grad, dL/d(initial x, v, C, F, params[, E, m])."""
    s = [p["x"], p["v"], p["C"], p["F"]]
    more = [p["params"], p["Ep"], p["mp"]]
    history = []
    with torch.no_grad():
        for n in range(T):
            history.append(s)
            s = list(_step64(p, n, *s, *more))
    if not grad:
        return s, None
    N, dim = p["x"].shape
    if mean_seed:
        gx = torch.zeros_like(p["x"])
        gx[:, 0] = 1.0 / N
        adj = [gx, torch.zeros_like(gx)]
    else:
        adj = [p["gx"], p["gv"]]
    adj += [torch.zeros_like(p["C"]), torch.zeros_like(p["F"])]
    total = [None if t is None else torch.zeros_like(t) for t in more]
    for n in range(T - 1, -1, -1):
        here = [t.detach().requires_grad_(True) for t in history.pop()]
        var = [None if t is None else t.detach().requires_grad_(True) for t in more]
        used = [t for t in var if t is not None]
        out = _step64(p, n, *here, *var)
        got = torch.autograd.grad(out, here + used, grad_outputs=adj, allow_unused=True)
        adj = [torch.zeros_like(h) if q is None else q for h, q in zip(here, got)]
        rest = list(got[4:])
        for i, t in enumerate(var):
            if t is not None:
                q = rest.pop(0)
                total[i] = total[i] + (0 if q is None else q)
    return s, adj + total


def exact(case, seed):
    kind, T = case["kind"], case["steps"]
    if kind == "batch":
        parts = [[] for _ in range(9)]
        for i, n, steps, grad in _batch_requests(case):
            final, grads = _reference(_inputs(case, seed * 1000 + i, particles=n), steps, grad, mean_seed=True)
            for k, t in enumerate(final + (grads[:5] if grad else [])):
                parts[k].append(t.reshape(-1))
        return [torch.cat(q) for q in parts]
    p = _inputs(case, seed)
    if kind == "noalloc":
        if case["walls"] == "slip":
            p["kind"], p["c"] = [1] * (2 * case["dim"]), [float(np.float32(0.2))] * (2 * case["dim"])
        return _reference(p, T, False)[0]
    if kind == "step":
        return _reference(p, T, False)[0]
    if kind == "fp64":
        p["C"] = torch.zeros_like(p["C"])
        final, grads = _reference(p, T, True)
        out = final + grads[:4] + [grads[4].reshape(case["hidden"], case["groups"])]
        return [t.cpu().numpy() for t in out]
    final, grads = _reference(p, T, True)
    if kind == "rollout":
        return final + grads[:5]
    return final + grads[:5] + [grads[5].cpu().numpy(), grads[6].cpu().numpy()]
