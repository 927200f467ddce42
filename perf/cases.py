"""Performance cases: what a user has this library compute, through its public
Python entry points, from the smallest calls to the largest.

Four kinds of work, as the README describes the library's use:

  force     one lattice: set up, march the whole protocol, read the force back
            (Solver.run, or compute_force with the handle made in the call);
  ensemble  many independent lattices in one batched run (Batch.run);
  predict   forces from the trained surrogate network (MLP.predict);
  train     fitting the surrogate network to lattice forces (Surrogate.fit).

Lattice sizes, wavelengths, radii and point counts are those of workloads.py,
of the driven-cavity test and of the README's benchmarks; the number of
periods is cut where the whole protocol would take seconds, keeping unsampled
and sampled periods in about the protocol's 2 : 1 to 3 : 1 proportion.

exact() computes the same results with plain torch in 64 bits: lattice steps
that collide whole fields and stream them by rolling, and the network without
any rounding of its operands.
"""
import math

import numpy as np
import torch

import paper_2404_02346_gb300 as wlb
from paper_2404_02346_gb300 import surrogate

P_A = 1e-3
C0 = 0.25
BOX = {"ka": (0.1, 1.2), "kz": (0.0, math.pi), "c_ratio": (0.8, 2.0)}
GOLDEN_TURN = 0.3819660112501051517954131656


def listed():
    return [
        # The 2D cylinder validation run in FP64 (128 x 128, 64 points, 20 periods,
        # the last 5 averaged): the smallest whole force evaluation, made from
        # scratch by one compute_force call, with the final fields read for a plot.
        dict(name="cylinder_2d_f64", kind="force", dim=2, nx=128, ny=128, nz=1, axis=1, wavelength=64, radius=8.0,
             points=64, periods=20, avg=5, precision="f64", driven=False, fresh=True, fields=False),
        # The driven cavity of the paper's results section in 2D (lambda = 400,
        # length lambda/2 + 3, 64-cell lateral box, R = 8, walls damped by 0.99),
        # FP64, with the pressure and velocity fields read back.
        dict(name="cavity_2d_f64", kind="force", dim=2, nx=64, ny=203, nz=1, axis=1, wavelength=400, radius=8.0,
             points=64, periods=6, avg=2, precision="f64", driven=True, fresh=False, fields=True),
        # A small 3D sphere on odd, ragged rows, full 30-period protocol: a quick
        # look at one object on a lattice nobody rounded up to a power of two.
        dict(name="sphere_odd_f32", kind="force", dim=3, nx=57, ny=45, nz=64, axis=2, wavelength=32, radius=5.0,
             points=500, periods=30, avg=10, precision="f32", driven=False, fresh=False, fields=True),
        # The paper's 3D cavity: 64 x 64 lateral box, lambda = 400.
        dict(name="cavity_3d_f32", kind="force", dim=3, nx=64, ny=64, nz=203, axis=2, wavelength=400, radius=8.0,
             points=1000, periods=2, avg=1, precision="f32", driven=True, fresh=False, fields=False),
        # The 256^3 sphere benchmark (lambda = 128, R = 16, 2000 points), FP32.
        dict(name="sphere_256_f32", kind="force", dim=3, nx=256, ny=256, nz=256, axis=2, wavelength=128, radius=16.0,
             points=2000, periods=3, avg=1, precision="f32", driven=False, fresh=False, fields=False),
        # The same with FP16 storage of the populations.
        dict(name="sphere_256_f16", kind="force", dim=3, nx=256, ny=256, nz=256, axis=2, wavelength=128, radius=16.0,
             points=2000, periods=3, avg=1, precision="f16", driven=False, fresh=False, fields=False),
        # One position of the 512^3 force-vs-position sweep (R = 24, 4096 points),
        # the largest lattice; a shorter wavelength keeps the periods short.
        dict(name="sphere_512_f32", kind="force", dim=3, nx=512, ny=512, nz=512, axis=2, wavelength=64, radius=24.0,
             points=4096, periods=3, avg=1, precision="f32", driven=False, fresh=False, fields=False),
        # 64 spheres of uneven lattice sizes run together.
        dict(name="ensemble_3d_f32", kind="ensemble", dim=3, count=64, edges="96,128,160", points=1000, periods=3,
             avg=1, precision="f32"),
        # 512 cylinders on 192 x 192 lattices: how the surrogate's training data are made.
        dict(name="ensemble_2d_f32", kind="ensemble", dim=2, count=512, edges="192", points=1000, periods=5, avg=2,
             precision="f32"),
        # The surrogate asked for a handful of configurations (an interactive
        # query or one iteration of an optimiser) and for a dense sweep.
        dict(name="predict_1000", kind="predict", n=1000),
        dict(name="predict_1m", kind="predict", n=1 << 20),
        # One epoch of fitting the surrogate to 20 000 lattice forces.
        dict(name="train_20000", kind="train", samples=20000, batch=512, epochs=1),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _width(rng, lo, hi):
    """A lattice extent: half of the time a multiple of 16, as most users round, else any."""
    n = _log_int(rng, lo, hi)
    return max(lo, 16 * ((n + 8) // 16)) if rng.random() < 0.5 else n


def _reach(radius, surface_radius):
    return max(math.sqrt(radius * radius + 80.0), surface_radius + 1.5) + 1.0


def _draw_force(rng, dim):
    driven = rng.random() < 0.3
    if dim == 2:
        precision = rng.choice(["f64", "f64", "f32", "f32", "f16"])
        nx = _width(rng, 32, 600)
        wavelength = 2 * _log_int(rng, 28 if driven else 12, 200 if driven else 100)
        ny, nz = wavelength // 2 + 3 if driven else wavelength * rng.randint(1, 3), 1
        span, points = min(nx, ny), _log_int(rng, 48, 1000)
    else:
        precision = rng.choice(["f32", "f32", "f32", "f16"])
        nx, ny = _width(rng, 32, 300), _width(rng, 32, 256)
        wavelength = 2 * _log_int(rng, 28 if driven else 12, 200 if driven else 64)
        ny_nz = wavelength // 2 + 3 if driven else wavelength * rng.randint(1, 3)
        nz = ny_nz if driven or ny_nz <= 256 else wavelength
        span, points = min(nx, ny, nz), _log_int(rng, 100, 2000)
    # the object, its band and the stencil fit half the box (clear of the walls)
    room = span / 2.0 - (3.5 if driven else 1.0)
    radius = math.floor(4 * min(rng.uniform(3.0, 16.0), math.sqrt(max(room * room - 81.0, 9.0)), room - 3.0)) / 4.0
    radius = max(radius, 1.0)
    period = int(wavelength / C0)
    budget = 8000 if dim == 2 else max(2 * period, min(3000, int(4e10 / (nx * ny * nz))))
    periods = max(2, min(30, budget // period))
    return dict(kind="force", dim=dim, nx=nx, ny=ny, nz=nz, axis=dim - 1, wavelength=wavelength, radius=radius,
                points=points, periods=periods, avg=max(1, periods // 3), precision=precision, driven=driven,
                fresh=rng.random() < 0.3, fields=nx * ny * nz < 300000 and rng.random() < 0.5)


def draw(rng):
    u = rng.random()
    if u < 0.25:
        return _draw_force(rng, 2)
    if u < 0.5:
        return _draw_force(rng, 3)
    if u < 0.6:
        edges = sorted({8 * rng.randint(6, 20) for _ in range(rng.randint(1, 3))})
        return dict(kind="ensemble", dim=3, count=_log_int(rng, 4, 48), edges=",".join(map(str, edges)),
                    points=_log_int(rng, 200, 1500), periods=3, avg=1, precision=rng.choice(["f32", "f32", "f16"]))
    if u < 0.75:
        edges = sorted({16 * rng.randint(4, 14) for _ in range(rng.randint(1, 2))})
        return dict(kind="ensemble", dim=2, count=_log_int(rng, 32, 512), edges=",".join(map(str, edges)),
                    points=_log_int(rng, 64, 1000), periods=rng.randint(3, 6), avg=2,
                    precision=rng.choice(["f32", "f32", "f16"]))
    if u < 0.9:
        return dict(kind="predict", n=_log_int(rng, 1, 1 << 20))
    return dict(kind="train", samples=_log_int(rng, 2500, 30000), batch=rng.choice([128, 256, 512, 1024, 2048]),
                epochs=rng.randint(1, 2))


# ---------------------------------------------------------------- inputs
def _problem(dim, n, axis, wavelength, radius, center, c_ratio, points, periods, avg, precision, driven=False):
    """A problem dictionary as Solver and Batch take it (lattice units)."""
    period = int(round(wavelength / C0))
    p = dict(dim=dim, n=tuple(n), wave_axis=axis, c0=C0, cp=c_ratio * C0, rho0=1.0, p_a=P_A,
             wavelength=float(wavelength), antinode=0.0,
             center=tuple(math.floor(c * 1024.0) / 1024.0 for c in center) + (0.0,) * (3 - len(center)),
             radius=float(radius), interface_d=4.0, surface_radius=float(radius) + (1.0 if driven else 0.0),
             n_surface=points, n_steps=periods * period, n_window=avg * period, period=period, precision=precision)
    if driven:
        p.update(boundary="driven", wall_damping=0.99, source_amplitude=P_A / C0 ** 2)
    return p


def _problems(case, seed):
    g = np.random.default_rng(seed)
    common = dict(points=case["points"], periods=case["periods"], avg=case["avg"], precision=case["precision"])
    dim = case["dim"]
    if case["kind"] == "force":
        n = (case["nx"], case["ny"], case["nz"])
        center = [n[a] / 2.0 + g.uniform(-0.5, 0.5) for a in range(dim)]
        ax, lam, R = case["axis"], case["wavelength"], case["radius"]
        if case["driven"]:  # an eighth of a wavelength from the source-side antinode, clear of the walls
            lo = 2.0 + _reach(R, R + 1.0)
            center[ax] = min(max(1.0 + lam / 8.0 + g.uniform(-2.0, 2.0), lo + 0.01), n[ax] - lo - 0.01)
        else:
            center[ax] = lam * g.uniform(0.08, 0.17)
        return [_problem(dim, n, ax, lam, R, center, g.uniform(1.15, 2.0), driven=case["driven"], **common)]
    edges = [int(e) for e in case["edges"].split(",")]
    out = []
    for i in range(case["count"]):
        edge = edges[int(g.integers(len(edges)))]
        lam = edge // 2
        z0 = lam * g.uniform(0.0, 0.5)
        R = math.floor(g.uniform(4.0, 12.0) * 1024.0) / 1024.0
        out.append(_problem(dim, (edge,) * dim + (1,) * (3 - dim), dim - 1, lam, R, (edge / 2.0,) * (dim - 1) + (z0,),
                            g.uniform(0.8, 2.0), **common))
    return out


def _features(n, seed):
    """n rows (k R, k z0, kappa~, c~) in the surrogate's box."""
    g = np.random.default_rng(seed)
    ka, kz, c = (g.uniform(*BOX[k], size=n) for k in ("ka", "kz", "c_ratio"))
    return np.stack([ka, kz, 1.0 / c ** 2, c], axis=1).astype(np.float32)


def _targets(x):
    """Normalised forces of about the lattice's shape: Wei's law with a finite-size term."""
    ka, kz, kappa = (x[:, i].astype(np.float64) for i in range(3))
    return ((1.0 - kappa) * np.sin(2.0 * kz) * (1.0 + 0.15 * ka ** 2)).astype(np.float32)


def _weights(seed):
    """A network's packed FP32 parameters, U(-1/sqrt(fan_in), 1/sqrt(fan_in)) per layer."""
    g = np.random.default_rng(seed + 1000003)
    parts = []
    for out, fan in ((256, 4), (256, 256), (256, 256), (1, 256)):
        a = 1.0 / math.sqrt(fan)
        parts += [g.uniform(-a, a, size=out * fan), g.uniform(-a, a, size=out)]
    return np.concatenate(parts).astype(np.float32)


def _box():
    s = BOX
    lo = np.array([s["ka"][0], s["kz"][0], 1.0 / s["c_ratio"][1] ** 2, s["c_ratio"][0]], dtype=np.float32)
    hi = np.array([s["ka"][1], s["kz"][1], 1.0 / s["c_ratio"][0] ** 2, s["c_ratio"][1]], dtype=np.float32)
    return lo, hi


def prepare(case, seed):
    kind = case["kind"]
    if kind == "force":
        p = _problems(case, seed)[0]
        return dict(kind=kind, problem=p, fields=case["fields"], solver=None if case["fresh"] else wlb.Solver(p))
    if kind == "ensemble":
        return dict(kind=kind, batch=wlb.Batch(_problems(case, seed)))
    if kind == "predict":
        lo, hi = _box()
        net = wlb.MLP(lo, hi)
        net.set_weights(_weights(seed))
        return dict(kind=kind, net=net, x=torch.from_numpy(_features(case["n"], seed)).cuda())
    x = _features(case["samples"], seed)
    return dict(kind=kind, surrogate=surrogate.Surrogate(BOX, batch_max=4096), x=x, t=_targets(x),
                epochs=case["epochs"], batch=case["batch"], seed=int(seed) & 0x7fffffff)


def run(state):
    kind = state["kind"]
    if kind == "force":
        s = state["solver"]
        if s is None and not state["fields"]:
            return dict(force=wlb.compute_force(state["problem"]))
        own = s is None
        if own:
            s = wlb.Solver(state["problem"])
        out = dict(force=s.run())
        out["history"] = s.force_history()
        if state["fields"]:
            out["p1"], out["u1"] = s.fields()
        if own:
            s.close()
        return out
    if kind == "ensemble":
        return dict(forces=state["batch"].run())
    if kind == "predict":
        y, inside = state["net"].predict(state["x"])
        return dict(y=y, inside=inside)
    sur = state["surrogate"]
    history = sur.fit(state["x"], state["t"], epochs=state["epochs"], batch=state["batch"], seed=state["seed"])
    return dict(history=history, weights=sur.net.get_weights())


# ---------------------------------------------------------------- work
def work(case):
    """Bytes: the state the call starts from and the results, each once (a
    lattice's populations and classes; everything between can stay on the
    chip).  Operations: the additions and multiplications of every cell
    update, or of the matrix products."""
    kind = case["kind"]
    if kind in ("force", "ensemble"):
        dim = case["dim"]
        q, ops = 2 * dim + 1, 12 if dim == 2 else 16
        size = {"f64": 8, "f32": 4, "f16": 2}[case["precision"]]
        if kind == "force":
            shapes = [((case["nx"], case["ny"], case["nz"]), case["wavelength"])]
            fields = 8 * (1 + dim) * case["nx"] * case["ny"] * case["nz"] if case["fields"] else 0
        else:
            edges = [int(e) for e in case["edges"].split(",")]
            shapes = [((edges[i % len(edges)],) * dim, edges[i % len(edges)] // 2) for i in range(case["count"])]
            fields = 0
        cells = [math.prod(n) for n, _ in shapes]
        steps = [case["periods"] * int(lam / C0) for _, lam in shapes]
        return dict(bytes=sum(cells) * (2 * q * size + 1) + fields + 24 * len(shapes),
                    flops=sum(c * s for c, s in zip(cells, steps)) * ops)
    weights = 4 * 256 + 256 * 256 * 2 + 256
    if kind == "predict":
        return dict(bytes=case["n"] * (16 + 4 + 1) + 4 * (weights + 769), flops=2 * weights * case["n"])
    steps = case["epochs"] * (case["samples"] // case["batch"])
    return dict(bytes=case["samples"] * 20 + 4 * (weights + 769), flops=6 * weights * case["batch"] * steps)


# ---------------------------------------------------------------- 64-bit results
def _kernel3(r):
    a = r.abs()
    inner = (1.0 + torch.sqrt((1.0 - 3.0 * r * r).clamp(min=0.0))) / 3.0
    outer = (5.0 - 3.0 * a - torch.sqrt((1.0 - 3.0 * (1.0 - a) ** 2).clamp(min=0.0))) / 6.0
    return torch.where(a <= 0.5, inner, torch.where(a <= 1.5, outer, torch.zeros_like(a)))


def _surface(p, dev):
    """Normals, element areas, stencil cell indices and kernel weights of one problem's surface."""
    N, R, dim, n = p["n_surface"], p["surface_radius"], p["dim"], p["n"]
    k = torch.arange(N, dtype=torch.float64, device=dev)
    nrm = torch.zeros(N, 3, dtype=torch.float64, device=dev)
    if dim == 2:
        t = 2.0 * math.pi * (2.0 * k + 1.0) / (2.0 * N)
        nrm[:, 0], nrm[:, 1] = torch.cos(t), torch.sin(t)
        dS = 2.0 * math.pi * R / N
    else:
        z = 1.0 - (2.0 * k + 1.0) / N
        rho = torch.sqrt(1.0 - z * z)
        t = 2.0 * math.pi * torch.frac(k * GOLDEN_TURN)
        nrm[:, 0], nrm[:, 1], nrm[:, 2] = rho * torch.cos(t), rho * torch.sin(t), z
        dS = 4.0 * math.pi * R * R / N
    X = torch.tensor(p["center"], dtype=torch.float64, device=dev) + R * nrm
    base = torch.floor(X + 0.5)
    off = torch.tensor([[dx, dy, dz] for dz in ((-1, 0, 1) if dim == 3 else (0,)) for dy in (-1, 0, 1)
                        for dx in (-1, 0, 1)], dtype=torch.float64, device=dev)
    c = base[:, None, :] + off[None]
    if dim == 2:
        c[..., 2] = 0.0
    w = torch.ones(c.shape[:2], dtype=torch.float64, device=dev)
    for a in range(dim):
        w = w * _kernel3(c[..., a] - X[:, None, a])
    c = c.long()
    idx = (torch.remainder(c[..., 2], n[2]) * n[1] + torch.remainder(c[..., 1], n[1])) * n[0] + \
        torch.remainder(c[..., 0], n[0])
    return nrm, dS, idx, w


def _sound_speed_sq(p, dev):
    q = -p["radius"] ** 2
    n = p["n"]
    for a, shape in zip(range(p["dim"]), ((1, 1, -1), (1, -1, 1), (-1, 1, 1))):
        d = torch.arange(n[a], dtype=torch.float64, device=dev) - p["center"][a]
        d = torch.where(d >= 0.5 * n[a], d - n[a], torch.where(d < -0.5 * n[a], d + n[a], d))
        q = q + (d * d).view(shape)
    c = p["cp"] + 0.5 * (p["c0"] - p["cp"]) * (1.0 + torch.tanh(q / p["interface_d"]))
    c = torch.where(q >= 20.0 * p["interface_d"], p["c0"], torch.where(q <= -20.0 * p["interface_d"], p["cp"], c))
    return (c * c).expand(n[2], n[1], n[0])


def _exact_lattices(problems):
    """Forces, per-period forces and final fields of problems on lattices of
    one size and wavelength: collide, apply the walls, stream by rolling."""
    p = problems[0]
    dev = "cuda" if torch.cuda.is_available() else "cpu"
    dim, n, ax, B = p["dim"], p["n"], p["wave_axis"], len(problems)
    T, rho0 = p["period"], p["rho0"]
    driven = p.get("boundary") == "driven"
    c2 = torch.stack([_sound_speed_sq(q, dev) for q in problems])  # [B, z, y, x]
    surf = [_surface(q, dev) for q in problems]
    nrm = torch.stack([s[0] for s in surf])
    dS = torch.tensor([s[1] for s in surf], dtype=torch.float64, device=dev)
    cells = n[0] * n[1] * n[2]
    idx = torch.stack([s[2] + i * cells for i, s in enumerate(surf)])
    w = torch.stack([s[3] for s in surf])
    wp = w * c2.reshape(-1)[idx]
    tdim = (3, 2, 1)  # tensor axis of x, y, z
    s = torch.arange(n[ax], dtype=torch.float64, device=dev)
    shape = [1, 1, 1, 1]
    shape[tdim[ax]] = -1
    p0 = (p["p_a"] * torch.cos(2.0 * math.pi * (s - p["antinode"]) / p["wavelength"])).view(shape)
    if driven:
        p0 = torch.zeros_like(p0)
    f = [(p0 / c2 * (1.0 - dim * c2)).clone()] + [(0.5 * p0).expand_as(c2).clone() for _ in range(2 * dim)]
    at = lambda i: tuple(i if d == tdim[ax] else slice(None) for d in range(4))  # noqa: E731
    lo, src, hi = at(0), at(1), at(n[ax] - 1)
    phi, amp = p.get("wall_damping", 0.0), p.get("source_amplitude", 0.0)
    n_free = p["n_steps"] - p["n_window"]
    sums, history = torch.zeros(B, p["n_surface"], 5, dtype=torch.float64, device=dev), []
    total = torch.zeros_like(sums)

    def force(a, count):
        a = a / count
        iso = a[..., 0] / (2.0 * rho0 * p["c0"] ** 2) - 0.5 * rho0 * a[..., 1]
        F = -(dS[:, None, None] * (iso[..., None] * nrm + rho0 * a[..., 2:5])).sum(1)
        if dim == 2:
            F[:, 2] = 0.0
        return F

    for t in range(p["n_steps"]):
        rho = f[0].clone()
        for i in range(1, 2 * dim + 1):
            rho += f[i]
        if t >= n_free:
            pk = (wp * rho.reshape(-1)[idx]).sum(-1)
            u = torch.zeros(B, p["n_surface"], 3, dtype=torch.float64, device=dev)
            for a in range(dim):
                J = f[1 + 2 * a].reshape(-1)[idx] - f[2 + 2 * a].reshape(-1)[idx]
                u[..., a] = (w * J).sum(-1) / rho0
            un = (u * nrm).sum(-1)
            sums += torch.stack([pk * pk, (u * u).sum(-1), u[..., 0] * un, u[..., 1] * un, u[..., 2] * un], dim=-1)
            if (t + 1 - n_free) % T == 0:
                history.append(force(sums, T))
                total += sums
                sums.zero_()
        if driven:
            edge = {k: [v[sl].clone() for v in f] for k, sl in (("lo", lo), ("src", src), ("hi", hi))}
        eq = c2 * rho
        f[0] = 2.0 * (rho - dim * eq) - f[0]
        for a in range(dim):
            f[1 + 2 * a], f[2 + 2 * a] = eq - f[2 + 2 * a], eq - f[1 + 2 * a]
        if driven:
            for name, sl, out in (("lo", lo, 2 + 2 * ax), ("hi", hi, 1 + 2 * ax)):
                e = edge[name]
                f[0][sl] = phi * e[0]
                for a in range(dim):
                    f[1 + 2 * a][sl] = 0.0 if 1 + 2 * a == out else phi * e[2 + 2 * a]
                    f[2 + 2 * a][sl] = 0.0 if 2 + 2 * a == out else phi * e[1 + 2 * a]
            r = amp * math.sin(2.0 * math.pi * (t % T) / T)
            e, cs = edge["src"], c2[src]
            f[0][src] = r * (1.0 - dim * cs)
            for a in range(dim):
                J = e[1 + 2 * a] - e[2 + 2 * a]
                f[1 + 2 * a][src] = 0.5 * (cs * r + J)
                f[2 + 2 * a][src] = 0.5 * (cs * r - J)
        for a in range(dim):
            f[1 + 2 * a] = torch.roll(f[1 + 2 * a], 1, tdim[a])
            f[2 + 2 * a] = torch.roll(f[2 + 2 * a], -1, tdim[a])
    rho = sum(f[1:], f[0].clone())
    u1 = [(f[1 + 2 * a] - f[2 + 2 * a]) / rho0 for a in range(dim)]
    F = force(total, p["n_window"])
    return F, torch.stack(history, 1), c2 * rho, u1


def _gelu(z):
    return 0.5 * z * (1.0 + torch.erf(z / math.sqrt(2.0)))


def _layers(w):
    out, o = [], 0
    for rows, fan in ((256, 4), (256, 256), (256, 256), (1, 256)):
        out.append((w[o:o + rows * fan].view(rows, fan), w[o + rows * fan:o + rows * fan + rows]))
        o += rows * fan + rows
    return out


def _network(w, x):
    lo, hi = (torch.from_numpy(v.astype(np.float64)).to(x.device) for v in _box())
    h = 2.0 * (x - lo) / (hi - lo) - 1.0
    layers = _layers(w)
    for W, b in layers[:-1]:
        h = _gelu(h @ W.t() + b)
    W, b = layers[-1]
    return (h @ W.t() + b)[:, 0]


def _mixer(seed, n):
    """n outputs of the SplitMix64 generator."""
    with np.errstate(over="ignore"):
        z = np.uint64(seed) + np.arange(1, n + 1, dtype=np.uint64) * np.uint64(0x9E3779B97F4A7C15)
        z = (z ^ (z >> np.uint64(30))) * np.uint64(0xBF58476D1CE4E5B9)
        z = (z ^ (z >> np.uint64(27))) * np.uint64(0x94D049BB133111EB)
    return z ^ (z >> np.uint64(31))


def _exact_train(case, seed):
    """The training run with unrounded products and activations."""
    dev = "cuda" if torch.cuda.is_available() else "cpu"
    s, n, batch = int(seed) & 0x7fffffff, case["samples"], case["batch"]
    x = _features(n, seed)
    t = torch.from_numpy(_targets(x).astype(np.float64)).to(dev)
    x = torch.from_numpy(x.astype(np.float64)).to(dev)
    sizes = [(256 * 4, 4), (256, 4), (65536, 256), (256, 256), (65536, 256), (256, 256), (256, 256), (1, 256)]
    u = (_mixer(s, sum(k for k, _ in sizes)) >> np.uint64(11)).astype(np.float64) / 9007199254740992.0
    a = np.concatenate([np.full(k, np.float64(np.float32(1.0) / np.sqrt(np.float32(fan)))) for k, fan in sizes])
    w = torch.from_numpy(((2.0 * u - 1.0) * a).astype(np.float32).astype(np.float64)).to(dev).requires_grad_(True)
    m1, m2 = torch.zeros_like(w), torch.zeros_like(w)
    lr, lr_final, step, history = 2e-3, 2e-5, 0, []
    mix = [int(v) for v in _mixer(s, case["epochs"] * (n - 1))]
    drawn = iter(mix)
    for ep in range(case["epochs"]):
        perm = list(range(n))
        for i in range(n - 1, 0, -1):
            j = next(drawn) % (i + 1)
            perm[i], perm[j] = perm[j], perm[i]
        perm = torch.tensor(perm, device=dev)
        rate = lr * (lr_final / lr) ** (ep / max(case["epochs"] - 1, 1))
        losses = []
        for k in range(n // batch):
            at = perm[k * batch:(k + 1) * batch]
            loss = ((_network(w, x[at]) - t[at]) ** 2).mean()
            g, = torch.autograd.grad(loss, w)
            losses.append(loss.detach())
            step += 1
            with torch.no_grad():
                m1.mul_(0.9).add_(0.1 * g)
                m2.mul_(0.999).add_(0.001 * g * g)
                w -= rate * (m1 / (1.0 - 0.9 ** step)) / (torch.sqrt(m2 / (1.0 - 0.999 ** step)) + 1e-8)
        history.append(torch.stack(losses).mean())
    return dict(history=torch.stack(history).cpu().numpy(), weights=w.detach().cpu().numpy())


def exact(case, seed):
    kind = case["kind"]
    if kind == "force":
        F, H, p1, u1 = _exact_lattices(_problems(case, seed))
        out = dict(force=F[0].cpu().numpy())
        if not (case["fresh"] and not case["fields"]):
            out["history"] = H[0].cpu().numpy()
        if case["fields"]:
            out["p1"], out["u1"] = p1[0].cpu().numpy(), torch.stack([v[0] for v in u1]).cpu().numpy()
        return out
    if kind == "ensemble":
        problems = _problems(case, seed)
        F = np.zeros((len(problems), 3))
        for n in sorted({q["n"] for q in problems}):
            at = [i for i, q in enumerate(problems) if q["n"] == n]
            F[at] = _exact_lattices([problems[i] for i in at])[0].cpu().numpy()
        return dict(forces=F)
    if kind == "predict":
        dev = "cuda" if torch.cuda.is_available() else "cpu"
        x = torch.from_numpy(_features(case["n"], seed)).to(dev)
        w = torch.from_numpy(_weights(seed).astype(np.float64)).to(dev)
        y = torch.cat([_network(w, part.double()) for part in x.split(1 << 16)])
        return dict(y=y, inside=None)
    return _exact_train(case, seed)
