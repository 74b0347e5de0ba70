"""What a user of this framework has it do, as cases that can be timed.

Every case is a part of a program that a user writes: a time loop on one grid, a sweep of
many small problems, a report, training and using a learned trace, a field that lives on the
host.  The sizes come from this repository's configurations, tests and benchmark.

A grid's time loop returns the 1 + dim planes that a user keeps (phi and its gradient, what
set_state takes back; the mixed derivatives are rebuilt from them) and goes on from where
it is at the next pass, except where a case is a whole run from given initial data.
"""
import math

import numpy as np
import torch

from paper_0905_3409_gb300 import gals, inputs

PI = math.pi


def listed():
    return [
        # the smallest work: a program that picks its own time step calls step() once per
        # step on the 64^2 grid of the convergence tests, and looks at all planes after 16
        dict(name="calls_64", kind="grid", nx=64, ny=64, nz=1, field="vortex2d", modes=0, layout="full",
             cross="central", trace="rk3", cfl=1.0, calls=16, steps=1, restart=False, planes=4, shape="round"),
        # the 64^2 single-vortex run of the paper's first test, whole: initial data in, 504
        # steps in one call, result out (the loop of every convergence study)
        dict(name="run_64", kind="grid", nx=64, ny=64, nz=1, field="vortex2d", modes=0, layout="full",
             cross="central", trace="rk3", cfl=1.0, calls=1, steps=504, restart=True, planes=3, shape="round"),
        # an everyday grid of odd, unequal sides in the compact layout: Zalesak's disk
        dict(name="slotted_1021x777", kind="grid", nx=1021, ny=777, nz=1, field="rotation", modes=0,
             layout="compact", cross="central", trace="rk3", cfl=1.0, calls=1, steps=100, restart=False, planes=3,
             shape="slotted"),
        # the headline grid: 4096^2 single vortex, 20 steps between two looks at the state
        dict(name="vortex_4096", kind="grid", nx=4096, ny=4096, nz=1, field="vortex2d", modes=0, layout="full",
             cross="central", trace="rk3", cfl=1.0, calls=1, steps=20, restart=False, planes=3, shape="round"),
        # the paper's 3D volume tables: 101^3, time steps of CFL 2
        dict(name="sphere_101", kind="grid", nx=101, ny=101, nz=101, field="deform3d", modes=0, layout="full",
             cross="central", trace="rk3", cfl=2.0, calls=1, steps=50, restart=False, planes=4, shape="round"),
        # the large 3D run: 512^3 deformation
        dict(name="deform_512", kind="grid", nx=512, ny=512, nz=512, field="deform3d", modes=0, layout="full",
             cross="central", trace="rk3", cfl=1.0, calls=1, steps=8, restart=False, planes=4, shape="round"),
        # many independent problems of uneven size, each with its own field and time step
        dict(name="batch_256", kind="batch", count=256, nmin=128, nmax=1024, modes=8, layout="full", steps=10),
        # a velocity that is costly to evaluate
        dict(name="waves_2048", kind="grid", nx=2048, ny=2048, nz=1, field="waves2d", modes=256, layout="full",
             cross="central", trace="rk3", cfl=1.0, calls=1, steps=2, restart=False, planes=3, shape="round"),
        # the learned trace in the time loop
        dict(name="learned_2048", kind="learned", n=2048, modes=16, steps=4),
        # fitting the learned trace: a stretch of its training
        dict(name="train_16384", kind="train", n=2048, modes=16, batch=16384, steps=50),
        # a report on a run: area, difference to a reference, normals and curvature at points
        dict(name="report_2048", kind="report", nx=2048, ny=2048, nz=1, q=4, points=200000),
        # a field that lives on the host, stepped through the device
        dict(name="host_2048", kind="host", nx=2048, ny=2048, nz=1, steps=4),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["grid2", "grid2", "grid2", "grid2", "grid3", "grid3", "batch", "waves", "learned", "train",
                       "report", "host"])
    if kind == "grid2":
        nx = _log(rng, 24, 4096)
        ny = max(24, min(4096, int(nx * rng.uniform(0.4, 1.6))))
        field = rng.choice(["vortex2d", "rotation", "fourier2d"])
        cross = rng.choice(["central", "central", "central", "cell"])
        steps = max(2, min(_log(rng, 2, 504), int(20 * 4096 ** 2 / (nx * ny))))
        calls = rng.choice([1, 1, 1, 4])
        return dict(kind="grid", nx=nx, ny=ny, nz=1, field=field, modes=16 if field == "fourier2d" else 0,
                    layout=rng.choice(["full", "full", "compact"]) if cross == "central" else "full", cross=cross,
                    trace=rng.choice(["rk3", "rk3", "rk3", "heun_psi", "euler"]), cfl=rng.choice([0.5, 1.0, 1.0, 2.0]),
                    calls=calls, steps=max(1, steps // calls), restart=rng.random() < 0.2, planes=3,
                    shape="slotted" if field == "rotation" and nx <= 1024 else "round")
    if kind == "grid3":
        nx = _log(rng, 16, 400)
        ny, nz = (max(16, min(400, int(nx * rng.uniform(0.6, 1.4)))) for _ in range(2))
        steps = max(2, min(_log(rng, 2, 100), int(4 * 400 ** 3 / (nx * ny * nz))))
        return dict(kind="grid", nx=nx, ny=ny, nz=nz, field=rng.choice(["deform3d", "deform3d", "rotation"]), modes=0,
                    layout=rng.choice(["full", "full", "compact"]), cross="central",
                    trace=rng.choice(["rk3", "rk3", "rk3", "heun_psi"]), cfl=rng.choice([0.5, 1.0, 1.0, 2.0]), calls=1,
                    steps=steps, restart=False, planes=4, shape="round")
    if kind == "batch":
        nmin = _log(rng, 32, 300)
        nmax = nmin + _log(rng, 16, 600)
        count = max(4, min(_log(rng, 8, 256), int(8e7 / nmax ** 2)))
        return dict(kind="batch", count=count, nmin=nmin, nmax=nmax, modes=rng.choice([4, 8, 16]),
                    layout=rng.choice(["full", "full", "compact"]), steps=_log(rng, 2, 20))
    if kind == "waves":
        n, modes = _log(rng, 100, 1500), _log(rng, 16, 512)
        return dict(kind="grid", nx=n, ny=max(64, n - rng.randrange(40)), nz=1, field="waves2d", modes=modes,
                    layout="full", cross="central", trace="rk3", cfl=rng.choice([0.5, 1.0]), calls=1,
                    steps=max(1, min(8, int(2 * 2048 ** 2 * 256 / (n * n * modes)))), restart=False, planes=3,
                    shape="round")
    if kind == "learned":
        return dict(kind="learned", n=_log(rng, 200, 2048), modes=16, steps=rng.choice([2, 4]))
    if kind == "train":
        return dict(kind="train", n=_log(rng, 256, 2048), modes=rng.choice([8, 16]), batch=_log(rng, 512, 16384),
                    steps=_log(rng, 10, 50))
    if kind == "report":
        if rng.random() < 0.5:
            nx = _log(rng, 100, 2048)
            return dict(kind="report", nx=nx, ny=max(64, int(nx * rng.uniform(0.5, 1.0))), nz=1,
                        q=rng.choice([2, 4, 8]), points=_log(rng, 1000, 200000))
        nx = _log(rng, 32, 160)
        return dict(kind="report", nx=nx, ny=max(32, int(nx * rng.uniform(0.6, 1.0))), nz=_log(rng, 32, 160),
                    q=rng.choice([2, 4]), points=_log(rng, 1000, 200000))
    nx = _log(rng, 512, 2048)
    return dict(kind="host", nx=nx, ny=max(256, int(nx * rng.uniform(0.5, 1.0))), nz=1, steps=rng.choice([1, 4]))


# ------------------------------------------------------------------ inputs

def _sizes(case):
    if "n" in case:
        return (case["n"], case["n"])
    return (case["nx"], case["ny"]) if case["nz"] == 1 else (case["nx"], case["ny"], case["nz"])


def _axes(n, dtype=torch.float64):
    """Coordinates of the nodes as broadcastable tensors, x last."""
    dim = len(n)
    out = []
    for d in range(dim):
        shape = [1] * dim
        shape[dim - 1 - d] = n[d]
        out.append((torch.arange(n[d], device="cuda", dtype=dtype) / (n[d] - 1)).reshape(shape))
    return out


def _round_state(n, center, r):
    """Signed distance to a circle or sphere and its gradient, FP32 planes on the GPU."""
    dx = [x - c for x, c in zip(_axes(n), center)]
    out = torch.empty((1 + len(n),) + tuple(reversed(n)), dtype=torch.float32, device="cuda")
    for k in range(out.shape[1]):  # by rows or levels, to keep the FP64 temporaries small
        d = [v if v.shape[0] == 1 else v[k:k + 1] for v in dx]
        rr = torch.sqrt(sum(v * v for v in d)).clamp_min(1e-30)
        out[0, k:k + 1] = rr - r
        for a, v in enumerate(d):
            out[1 + a, k:k + 1] = v / rr
    return out


def _round_state_small(n, center, r):
    """The same at once, for grids whose temporaries fit."""
    dx = [x - c for x, c in zip(_axes(n), center)]
    rr = torch.sqrt(sum(v * v for v in dx)).clamp_min(1e-30)
    return torch.stack([rr - r] + [(v / rr).expand(rr.shape) for v in dx]).float()


def _shape_of(case, seed, extra=0):
    """Where this seed's circle or sphere lies."""
    rng = np.random.default_rng([seed, extra])
    dim = len(_sizes(case))
    if dim == 2:
        return (0.5 + rng.uniform(-0.05, 0.05), 0.75 + rng.uniform(-0.05, 0.05)), 0.15 + rng.uniform(-0.03, 0.03)
    return tuple(0.35 + rng.uniform(-0.05, 0.05, 3)), 0.15 + rng.uniform(-0.03, 0.03)


def _initial(case, seed, extra=0):
    n = _sizes(case)
    c, r = _shape_of(case, seed, extra)
    if case.get("shape") == "slotted":
        return torch.from_numpy(inputs.slotted_disk_sdf(n, center=c, r=r, slot_top=c[1] + 0.1)[:3].astype(np.float32)).cuda()
    return (_round_state if math.prod(n) > 3e7 else _round_state_small)(n, c, r)


def _modes(case):
    """The field is part of the program, not of the data: it does not change with the seed."""
    if case.get("field") == "waves2d":
        return inputs.wave_modes(case["modes"])
    return inputs.fourier_modes(case["modes"], periodic=True) if case.get("modes") else None


def _speed(case, modes):
    field = case.get("field", "vortex2d" if case["kind"] == "host" else "fourier2d")
    if field == "waves2d":  # sampled: the sum of the amplitudes is far above the field's speed
        x, y = _axes((65, 65))
        m = torch.tensor(modes, device="cuda")[:, :, None, None]
        best = 0.0
        for k in range(8):
            c = m[:, 0] * torch.cos(2 * PI * m[:, 4] * k / 8 + m[:, 5]) * torch.cos(m[:, 1] * x + m[:, 2] * y + m[:, 3])
            best = max(best, (m[:, 2] * c).sum(0).abs().max().item(), (m[:, 1] * c).sum(0).abs().max().item())
        return 1.1 * best
    if field == "fourier2d":
        return inputs.fourier_speed_bound(modes)
    return {"vortex2d": 1.0, "rotation": PI, "deform3d": 2.0}[field]


def _dt(case, modes):
    return case.get("cfl", 1.0) / (max(_sizes(case)) - 1) / _speed(case, modes)


def _dts(case, dt):
    """The time step of each call: a program that picks its own varies it a little."""
    return [dt * (1.0 - 0.02 * (k % 3)) for k in range(case["calls"])]


T2, T3, OMEGA = 8.0, 3.0, 2 * PI  # modulation periods and angular speed of the tests


def _velocity(case, modes, **kw):
    field = case.get("field", "vortex2d" if case["kind"] == "host" else "fourier2d")
    return gals.Velocity(field, trace=kw.pop("trace", case.get("trace", "rk3")), T=T3 if field == "deform3d" else T2,
                         omega=OMEGA, center=(0.5, 0.5, 0.5), modes=modes, **kw)


def _batch_parts(case, seed):
    rng = np.random.default_rng([seed, 7])
    shape = np.random.default_rng([case["count"], case["nmin"], case["nmax"]])  # the program's own sizes and fields
    parts = []
    for _ in range(case["count"]):
        n = int(shape.integers(case["nmin"], case["nmax"] + 1))
        modes = inputs.fourier_modes(case["modes"], seed=int(shape.integers(1 << 31)))
        parts.append(dict(n=(n, n), modes=modes, dt=1.0 / (n - 1) / inputs.fourier_speed_bound(modes),
                          center=tuple(rng.uniform(0.3, 0.7, 2)), r=rng.uniform(0.08, 0.2)))
    return parts


def _points(case, seed):
    """Points in a band around this seed's circle or sphere, where a user asks for curvature."""
    c, r = _shape_of(case, seed)
    g = torch.Generator(device="cuda").manual_seed(seed)
    d = torch.randn((case["points"], len(c)), generator=g, device="cuda", dtype=torch.float64)
    band = r * (0.8 + 0.4 * torch.rand((case["points"], 1), generator=g, device="cuda", dtype=torch.float64))
    return torch.tensor(c, device="cuda", dtype=torch.float64) + d / d.norm(dim=1, keepdim=True) * band


_fitted = {}


def _fit(case):
    """Weights of the learned trace for the case's field and time step, fitted once: flat
    FP32 parameters (per layer W, then b) and the output scales, as set_params takes them."""
    key = (case["n"], case["modes"])
    if key in _fitted:
        return _fitted[key]
    modes = _modes(case)
    dt, h = _dt(case, modes), 1.0 / (case["n"] - 1)
    g = torch.Generator(device="cuda").manual_seed(5)
    X = torch.rand((1 << 18, 3), generator=g, device="cuda", dtype=torch.float64)
    vel = _field64("fourier2d", modes)
    out = []
    for x in X.split(1 << 15):
        d, J = _trace64("rk3", vel, [x[:, 0], x[:, 1]], x[:, 2], dt)
        out.append(torch.stack([d[0] / h, d[1] / h, (J[0][0] - 1) / dt, J[0][1] / dt, J[1][0] / dt, (J[1][1] - 1) / dt], 1))
    Y = torch.cat(out)
    scales = Y.square().mean(0).sqrt()
    X, Y = (2 * X - 1).float(), (Y / scales).float()
    ws = []
    for k, (i, o) in enumerate([(3, 128), (128, 128), (128, 128), (128, 128), (128, 6)]):
        a = 4.0 if k == 0 else math.sqrt(6.0 / (i + o))
        w = (2 * torch.rand((o, i), generator=g, device="cuda") - 1) * a
        b = (2 * torch.rand((o,), generator=g, device="cuda") - 1) * (4.0 if k == 0 else 0.0)
        ws += [w.requires_grad_(), b.requires_grad_()]
    opt = torch.optim.Adam(ws, lr=1e-3, fused=True)
    total = 2000
    for it in range(total):
        opt.param_groups[0]["lr"] = 1e-5 + 0.5 * (2e-3 - 1e-5) * (1 + math.cos(PI * it / total))
        at = it % 16 * 16384
        loss = (_mlp(ws, X[at:at + 16384]) - Y[at:at + 16384]).square().mean()
        opt.zero_grad(set_to_none=True)
        loss.backward()
        opt.step()
    _fitted[key] = (torch.cat([w.detach().reshape(-1) for w in ws]).cpu().numpy(), scales.float().cpu().numpy())
    return _fitted[key]


def _mlp(ws, x):
    for k in range(0, 8, 2):
        x = torch.nn.functional.silu(torch.nn.functional.linear(x, ws[k], ws[k + 1]))
    return torch.nn.functional.linear(x, ws[8], ws[9])


# ------------------------------------------------------------------ the cases

def prepare(case, seed):
    s = dict(case=case, kind=case["kind"])
    if case["kind"] == "batch":
        parts = _batch_parts(case, seed)
        b = gals.Batch([p["n"] for p in parts], layout=case["layout"])
        for k, p in enumerate(parts):
            b.set_state(k, _round_state_small(p["n"], p["center"], p["r"]).cpu().numpy(), recon=True)
        s["vels"] = [gals.Velocity("fourier2d", modes=p["modes"]) for p in parts]
        s["dts"] = [p["dt"] for p in parts]
        b.autotune(s["vels"], s["dts"], trial_steps=3)
        # where the states go on the device: phi and its gradient of each problem, one after the other
        sizes = [p["n"][0] * p["n"][1] for p in parts]
        s["out"] = torch.empty(3 * sum(sizes), device="cuda")
        at, s["ptrs"] = 0, []
        for m in sizes:
            s["ptrs"].append((gals.ctypes.c_void_p * 3)(*[s["out"].data_ptr() + 4 * (at + p * m) for p in range(3)]))
            at += 3 * m
        s["b"] = b
        return s
    if case["kind"] == "train":
        modes = _modes(case)
        s.update(S=gals.Surrogate(seed=seed + 1), vel=_velocity(case, modes), dt=_dt(case, modes), h=1.0 / (case["n"] - 1),
                 seed=seed)
        return s
    n, modes = _sizes(case), _modes(case)
    if case["kind"] == "report":
        s["g"], s["ref"] = gals.Grid(n), gals.Grid(n)
        s["g"].set_state(_initial(case, seed), recon=True)
        s["ref"].set_state(_initial(case, seed, 1), recon=True)
        s["points"] = _points(case, seed)
        return s
    if case["kind"] == "host":
        n2 = _initial(case, seed)
        full = torch.cat([n2, torch.zeros_like(n2[:1])])
        s.update(g=gals.Grid(n), vel=_velocity(case, modes), dt=_dt(case, modes), t=0.0)
        s["bufs"] = [torch.empty(full.shape, pin_memory=True) for _ in range(2)]
        s["bufs"][0].copy_(full)
        s["arrays"] = [b.numpy() for b in s["bufs"]]
        return s
    s["g"] = gals.Grid(n, layout=case.get("layout", "full"), cross=case.get("cross", "central"))
    s["initial"] = _initial(case, seed)
    s["g"].set_state(s["initial"], recon=True)
    s["dt"] = _dt(case, modes)
    if case["kind"] == "learned":
        params, scales = _fit(case)
        s["S"] = gals.Surrogate(seed=1)
        s["S"].set_params(params, scales)
        s["S"].bind(_velocity(case, modes), s["dt"], 1.0 / (case["n"] - 1))
        s["vel"] = _velocity(case, modes, trace="surrogate", surrogate=s["S"])
        planes = 3
    else:
        s["vel"] = _velocity(case, modes)
        s["dts"] = _dts(case, s["dt"])
        planes = case["planes"]
        if not case["restart"]:
            s["initial"] = None
    s["out"] = torch.empty((planes,) + tuple(reversed(n)), device="cuda")
    return s


def run(s):
    case, kind = s["case"], s["kind"]
    if kind == "grid":
        g = s["g"]
        if case["restart"]:
            g.set_state(s["initial"], recon=True)
        for dt in s["dts"]:
            g.step(s["vel"], dt, case["steps"])
        return g.read_state(out=s["out"], nfields=s["out"].shape[0])
    if kind == "learned":
        s["g"].step(s["vel"], s["dt"], case["steps"])
        return s["g"].read_state(out=s["out"], nfields=3)
    if kind == "batch":
        s["b"].step(s["vels"], s["dts"], case["steps"])
        for k, p in enumerate(s["ptrs"]):
            gals._bcheck(gals.lib().gals_batch_read_state(s["b"]._h, k, p, 3, gals.MEM_DEVICE), s["b"]._h)
        return s["out"]
    if kind == "train":
        r = s["S"].train(s["vel"], s["dt"], s["h"], steps=case["steps"], batch=case["batch"], seed=s["seed"])
        params, scales = s["S"].get_params()
        return dict(params=params, scales=scales, loss=np.array([r["initial_loss"], r["final_loss"]], np.float32))
    if kind == "report":
        d = s["g"].diagnostics(q=case["q"], reference=s["ref"])
        H, normal, kappa = s["g"].eval_points(s["points"])
        return dict(d, H=H, normal=normal, kappa=kappa)
    a, b = s["arrays"]
    for _ in range(case["steps"]):  # each step's output is the next step's input
        s["g"].step_host(s["vel"], s["dt"], s["t"], a, out=b, wait=False)
        s["t"] += s["dt"]
        a, b = b, a
    s["g"].synchronize()
    s["arrays"] = [a, b]
    return a[:3]


def work(case):
    """Bytes: the phi and gradient planes in and out at every step (a report: its state and
    reference once; training: the samples' weights and targets).  Operations: those of the
    formulas per node, mode or sample."""
    kind = case["kind"]
    if kind == "train":
        per = 3 * 2 * 50304 + 32 * 4 * (case["modes"] * 30 + 40)
        return dict(bytes=case["steps"] * (case["batch"] * 36 + 4 * 50822 * 7), flops=case["steps"] * case["batch"] * per)
    if kind == "batch":
        shape = np.random.default_rng([case["count"], case["nmin"], case["nmax"]])
        nodes = 0
        for _ in range(case["count"]):
            nodes += int(shape.integers(case["nmin"], case["nmax"] + 1)) ** 2
            shape.integers(1 << 31)
        return dict(bytes=nodes * case["steps"] * 24, flops=nodes * case["steps"] * 500)
    n = _sizes(case)
    nodes = math.prod(n)
    if kind == "report":
        return dict(bytes=nodes * 2 * 4 * 2 ** len(n) + case["points"] * (8 + 4) * (len(n) + 1), flops=nodes * 20)
    steps = case["steps"] * case.get("calls", 1)
    per = 280 if len(n) == 2 else 800
    if kind == "learned":
        per = 100608 + 100
    elif case.get("field") == "waves2d":
        per += 3 * 20 * case["modes"]
    elif case.get("field") == "fourier2d":
        per += 220
    return dict(bytes=nodes * steps * 8 * (1 + len(n)), flops=nodes * steps * per)


# ------------------------------------------------------------------ the same in 64 bits

def _field64(field, modes=None):
    """v(x, t) and its Jacobian: x a list of tensors, t a number or a tensor."""
    cos, sin = torch.cos, torch.sin

    def cosn(v):
        return torch.cos(v) if torch.is_tensor(v) else math.cos(v)

    def vortex(x, t):
        c = cosn(PI * t / T2)
        sx, sy, s2x, s2y = sin(PI * x[0]), sin(PI * x[1]), sin(2 * PI * x[0]), sin(2 * PI * x[1])
        d00 = -c * PI * s2x * s2y
        return [-c * sx * sx * s2y, c * s2x * sy * sy], [[d00, -2 * PI * c * sx * sx * cos(2 * PI * x[1])],
                                                       [2 * PI * c * cos(2 * PI * x[0]) * sy * sy, -d00]]

    def rotation(x, t):
        z = torch.zeros_like(x[0] + x[-1])
        v = [z - OMEGA * (x[1] - 0.5), z + OMEGA * (x[0] - 0.5)] + [z] * (len(x) - 2)
        D = [[z for _ in x] for _ in x]
        D[0][1], D[1][0] = z - OMEGA, z + OMEGA
        return v, D

    def deform(x, t):
        c = cosn(PI * t / T3)
        s, s2, c2 = [sin(PI * a) ** 2 for a in x], [sin(2 * PI * a) for a in x], [cos(2 * PI * a) for a in x]
        v = [2 * c * s[0] * s2[1] * s2[2], -c * s2[0] * s[1] * s2[2], -c * s2[0] * s2[1] * s[2]]
        q = c * PI * s2[0] * s2[1] * s2[2]
        return v, [[2 * q, 4 * PI * c * s[0] * c2[1] * s2[2], 4 * PI * c * s[0] * s2[1] * c2[2]],
                   [-2 * PI * c * c2[0] * s[1] * s2[2], -q, -2 * PI * c * s2[0] * s[1] * c2[2]],
                   [-2 * PI * c * c2[0] * s2[1] * s[2], -2 * PI * c * s2[0] * c2[1] * s[2], -q]]

    def waves(x, t):  # v = (-Psi_y, Psi_x), wave by wave
        u = v = xx = xy = yy = 0.0
        for a, kx, ky, ph, nn, chi in np.asarray(modes, dtype=np.float64).tolist():
            th = kx * x[0] + ky * x[1] + ph
            a = a * cosn(2 * PI * nn * t + chi)
            ac, as_ = a * cos(th), -a * sin(th)
            u, v = u - ky * ac, v + kx * ac
            xx, xy, yy = xx + kx * kx * as_, xy + kx * ky * as_, yy + ky * ky * as_
        return [u, v], [[-xy, -yy], [xx, xy]]

    def fourier(x, t):  # v = (-Psi_y, Psi_x), modes of the same k, l together
        A = {}
        for a, k, l, nn, chi in np.asarray(modes, dtype=np.float64).tolist():
            A[k, l] = A.get((k, l), 0.0) + a * cosn(2 * PI * nn * t + chi)
        u = v = xx = xy = yy = 0.0
        Y = {l: (sin(l * PI * x[1]), l * PI * cos(l * PI * x[1])) for l in {l for _, l in A}}
        for k in {k for k, _ in A}:
            f = sum(a * Y[l][0] for (kk, l), a in A.items() if kk == k)
            fy = sum(a * Y[l][1] for (kk, l), a in A.items() if kk == k)
            fyy = sum(-a * (l * PI) ** 2 * Y[l][0] for (kk, l), a in A.items() if kk == k)
            s, c = sin(k * PI * x[0]), k * PI * cos(k * PI * x[0])
            u, v = u - s * fy, v + c * f
            xx, xy, yy = xx - (k * PI) ** 2 * s * f, xy + c * fy, yy + s * fyy
        return [u, v], [[-xy, -yy], [xx, xy]]

    return {"vortex2d": vortex, "rotation": rotation, "deform3d": deform, "waves2d": waves,
            "fourier2d": fourier}[field]


def _matmul(A, B):
    r = range(len(A))
    return [[sum(A[i][k] * B[k][j] for k in r) for j in r] for i in r]


def _lin(c, A, B=None, w=0.0):
    """c I + w A (+ w B), as nested lists."""
    r = range(len(A))
    return [[(c if i == j else 0.0) + w * (A[i][j] + (B[i][j] if B else 0.0)) for j in r] for i in r]


def _trace64(trace, vel, x, t, dt):
    """Displacement of the foot at t of the characteristic through x at t + dt, and the
    Jacobian of that map: forward Euler, or the Shu-Osher form of third order."""
    a, A = vel(x, t + dt)
    if trace == "euler":
        return [-dt * v for v in a], _lin(1.0, A, w=-dt)
    b, B = vel([p - dt * v for p, v in zip(x, a)], t)
    M = _matmul(B, _lin(1.0, A, w=-dt))
    c, C = vel([p - dt / 4 * (v + w) for p, v, w in zip(x, a, b)], t + dt / 2)
    N = _matmul(C, _lin(1.0, A, M, -dt / 4))
    J = _lin(1.0, A, M, -dt / 6)
    r = range(len(x))
    return [-dt * (a[i] / 6 + b[i] / 6 + 2 * c[i] / 3) for i in r], [[J[i][j] - 2 * dt / 3 * N[i][j] for j in r] for i in r]


def _diff(u, axis, h):
    """Central difference along an axis, of second order and one-sided at the ends."""
    u = u.movedim(axis, -1)
    d = torch.empty_like(u)
    d[..., 1:-1] = (u[..., 2:] - u[..., :-2]) / (2 * h)
    d[..., 0] = (-3 * u[..., 0] + 4 * u[..., 1] - u[..., 2]) / (2 * h)
    d[..., -1] = (3 * u[..., -1] - 4 * u[..., -2] + u[..., -3]) / (2 * h)
    return d.movedim(-1, axis)


def _planes64(core, h):
    """All planes by the exponents of their derivative, from phi and its gradient."""
    dim = len(h)
    P = {(0,) * dim: core[0]}
    for a in range(dim):
        P[tuple(int(b == a) for b in range(dim))] = core[1 + a]
    if dim == 2:
        P[1, 1] = _diff(core[2], -1, h[0])
    else:
        P[1, 1, 0], P[1, 0, 1] = _diff(core[2], -1, h[0]), _diff(core[3], -1, h[0])
        P[0, 1, 1] = _diff(core[3], -2, h[1])
        P[1, 1, 1] = _diff(P[0, 1, 1], -1, h[0])
    return P


def _weights64(xi, h):
    """Weights of (value 0, value 1, slope 0, slope 1) for derivatives 0, 1 and 2."""
    o = 1 - xi
    return [(o * o * (1 + 2 * xi), xi * xi * (3 - 2 * xi), h * xi * o * o, -h * xi * xi * o),
            (-6 * xi * o / h, 6 * xi * o / h, o * (1 - 3 * xi), xi * (3 * xi - 2)),
            ((12 * xi - 6) / h ** 2, (6 - 12 * xi) / h ** 2, (6 * xi - 4) / h, (6 * xi - 2) / h)]


def _hermite64(P, n, h, cell, xi, orders, per_cell=False):
    """The interpolant's derivatives at local coordinates xi of the cells, axis by axis."""
    dim = len(n)
    W = [_weights64(x, hh) for x, hh in zip(xi, h)]
    flat = {a: p.reshape(-1) for a, p in P.items()}
    stride = [1, n[0], n[0] * n[1]]
    base = sum(c * s for c, s in zip(cell, stride))
    got = {}

    def corner(c, a):
        if per_cell and a == (1, 1):  # phi_xy from the cell's own four edges
            gx, gy = (lambda i, j: corner((i, j), (1, 0))), (lambda i, j: corner((i, j), (0, 1)))
            e = [(gx(i, 1) - gx(i, 0)) / h[1] for i in (0, 1)]
            f = [(gy(1, j) - gy(0, j)) / h[0] for j in (0, 1)]
            return 0.75 * (e[c[0]] + f[c[1]]) - 0.25 * (e[1 - c[0]] + f[1 - c[1]])
        return flat[a][base + sum(i * s for i, s in zip(c, stride))]

    def reduced(axis, c, a, o):
        key = (axis, c, a, o)
        if key not in got:
            if axis == 0:
                got[key] = corner(c, a)
            else:
                w = W[axis - 1][o[-1]]
                got[key] = sum(w[2 * s + e] * reduced(axis - 1, (e,) + c, (s,) + a, o[:-1]) for e in (0, 1) for s in (0, 1))
        return got[key]

    return [reduced(dim, (), (), o) for o in orders]


def _locate64(x, n, h):
    cell, xi = [], []
    for p, m, hh in zip(x, n, h):
        p = p.clamp(0.0, 1.0)
        c = torch.floor(p / hh).long().clamp(0, m - 2)
        cell.append(c)
        xi.append(p / hh - c)
    return cell, xi


def _first(dim):
    return [tuple(int(a == b) for b in range(dim)) for a in range(dim)]


def _step64(P, n, t, dt, case, vel, given=None):
    """phi and its gradient after one step of the whole grid, by slabs along the last axis."""
    dim, h = len(n), [1.0 / (m - 1) for m in n]
    ax, out = _axes(n), torch.empty((1 + dim,) + P[(0,) * dim].shape, device="cuda", dtype=torch.float64)
    slab = max(1, int(6e6 * n[-1] / math.prod(n)))
    for k in range(0, n[-1], slab):
        x = [a if a.shape[0] == 1 else a[k:k + slab] for a in ax]
        full = torch.broadcast_shapes(*[a.shape for a in x])
        x = [a.expand(full) for a in x]
        d, J = given(x, t) if given else _trace64(case.get("trace", "rk3"), vel, x, t, dt)
        foot = [p + q for p, q in zip(x, d)]
        cell, xi = _locate64(foot, n, h)
        H, *g = _hermite64(P, n, h, cell, xi, [(0,) * dim] + _first(dim), case.get("cross") == "cell")
        if case.get("trace") == "heun_psi":
            Df, Dn = vel(foot, t)[1], vel(x, t + dt)[1]
            r = range(dim)
            k1 = [-sum(Df[b][a] * g[b] for b in r) for a in r]
            ps = [g[a] + dt * k1[a] for a in r]
            g = [g[a] + 0.5 * dt * (k1[a] - sum(Dn[b][a] * ps[b] for b in r)) for a in r]
        else:
            g = [sum(J[b][a] * g[b] for b in range(dim)) for a in range(dim)]
        out[0, k:k + slab] = H
        for a in range(dim):
            out[1 + a, k:k + slab] = g[a]
    return out


def exact(case, seed):
    kind = case["kind"]
    if kind == "train":
        return None  # BF16 operands and a few thousand steps of a descent: no value to compare with
    if kind == "batch":
        if case["count"] * case["nmax"] ** 2 * case["steps"] > 3e9:
            return None
        out = []
        for p in _batch_parts(case, seed):
            core, vel = _round_state_small(p["n"], p["center"], p["r"]).double(), _field64("fourier2d", p["modes"])
            for k in range(case["steps"]):
                core = _step64(_planes64(core, [1.0 / (m - 1) for m in p["n"]]), p["n"], k * p["dt"], p["dt"], {}, vel)
            out.append(core.reshape(-1))
        return torch.cat(out)
    n, modes = _sizes(case), _modes(case)
    h = [1.0 / (m - 1) for m in n]
    core = _initial(case, seed).double()
    if kind == "report":
        return _report64(case, seed, core, n, h)
    field = case.get("field", "vortex2d" if kind == "host" else "fourier2d")
    vel, dt, given, t = _field64(field, modes), _dt(case, modes), None, 0.0
    dts = _dts(case, dt) if kind == "grid" else [dt]
    if kind == "learned":
        params, scales = _fit(case)
        ws, at = [], 0
        for i, o in [(3, 128), (128, 128), (128, 128), (128, 128), (128, 6)]:
            for shape in ((o, i), (o,)):
                ws.append(torch.from_numpy(params[at:at + math.prod(shape)]).cuda().double().reshape(shape))
                at += math.prod(shape)
        sc = torch.from_numpy(scales).cuda().double()

        def given(x, t):
            ph = torch.full_like(x[0], 2 * (t - math.floor(t)) - 1).reshape(-1)
            X = torch.stack([2 * x[0].reshape(-1) - 1, 2 * x[1].reshape(-1) - 1, ph], 1)
            y = [torch.cat(v).reshape(x[0].shape) for v in zip(*[(_mlp(ws, q) * sc).unbind(1) for q in X.split(1 << 20)])]
            return [y[0] * h[0], y[1] * h[1]], [[1 + dt * y[2], dt * y[3]], [dt * y[4], 1 + dt * y[5]]]

    for d in dts:
        for k in range(case["steps"]):
            P = _planes64(core, h)
            if kind == "host" and k == 0:
                P[1, 1] = torch.zeros_like(core[0])  # as it is given
            core = _step64(P, n, t, d, case, vel, given)
            t += d
    if case.get("planes") == 4 and len(n) == 2:
        return torch.cat([core, _planes64(core, h)[1, 1][None]])
    return core


def _report64(case, seed, core, n, h):
    dim, q = len(n), case["q"]
    ref = _initial(case, seed, 1).double()
    P, R = _planes64(core, h), _planes64(ref, h)
    nneg = nsym = 0
    cells = [torch.arange(m - 1, device="cuda").reshape([-1 if a == dim - 1 - d else 1 for a in range(dim)]) for d, m in enumerate(n)]
    full = torch.broadcast_shapes(*[c.shape for c in cells])
    cells = [c.expand(full) for c in cells]
    for s in range(q ** dim):
        xi = [torch.full((1,) * dim, (s // q ** d % q + 0.5) / q, device="cuda", dtype=torch.float64) for d in range(dim)]
        neg = [_hermite64(S, n, h, cells, xi, [(0,) * dim])[0] < 0 for S in (P, R)]
        nneg += int(neg[0].sum())
        nsym += int((neg[0] != neg[1]).sum())
    unit = math.prod(h) / q ** dim
    x = _points(case, seed)
    cell, xi = _locate64(list(x.unbind(1)), n, h)
    first = _first(dim)
    second = [[tuple(a + b for a, b in zip(u, v)) for v in first] for u in first]
    got = _hermite64(P, n, h, cell, xi, [(0,) * dim] + first + sum(second, []))
    H, g, D = got[0], got[1:1 + dim], got[1 + dim:]
    norm = torch.sqrt(sum(v * v for v in g))
    tr = sum(D[a * dim + a] for a in range(dim))
    gDg = sum(g[a] * D[a * dim + b] * g[b] for a in range(dim) for b in range(dim))
    d = core - ref
    return dict(t=0.0, steps=None, samples=None, n_negative=None, measure_negative=nneg * unit, n_symdiff=None,
                measure_symdiff=nsym * unit, emax_phi=d[0].abs().max().item(), emax_psi=d[1:].abs().max().item(),
                l2_phi=math.sqrt(d[0].square().sum().item() * math.prod(h)), nonfinite=None, H=H,
                normal=torch.stack([v / norm for v in g], 1), kappa=(norm ** 2 * tr - gDg) / norm ** 3)
