"""The work that users of this framework have it do, as cases that can be timed and checked.

A case is a dict of plain values; `op` names the entry point:
  project   Plan.project: one pressure correction (transfer, divergence, solve, gradient)
  ib        Plan.project_ib: one time step of the immersed-boundary force iteration
  step      Momentum.predict, then Plan.project: one AB2 time step
  batch     project_batch: uneven 2D problems in one call
  serve     Batcher.launch: the requests that wait together in the request loop, 2D and 3D
  poisson   GridPlan.solve_poisson: the grid solve alone
Every case writes into output arrays that the caller keeps, as a time-stepping program does.
"""
import dataclasses
import math

import numpy as np
import torch

from paper_2304_14690_gb300 import pc
from paper_2304_14690_gb300 import workloads as wl

BETA, EPS, SUPPORT = 1.5, 6.3, 3.0      # workloads.Problem's defaults


def listed():
    return [
        # the smallest call: a periodic box without obstacles, plain FP64 (launches and latency)
        dict(name="taylor_green_64_fp64", op="project", geometry="taylor_green", dim=2, n0=64, n1=64, precision="fp64"),
        # the smallest request of the stream: inflow/outflow, walls and one cylinder
        dict(name="request_128_mixed", op="project", geometry="box", dim=2, n0=128, n1=128, bc="ID,WW",
             precision="mixed", obstacles=1),
        # the paper's cylinder in a periodic box (400 x 400, a length with factors of 5), with the
        # force of the previous pass
        dict(name="periodic_400_mixed", op="project", geometry="box", dim=2, n0=400, n1=400, bc="PP,PP",
             precision="mixed", obstacles=1, force=True),
        # the channel with a cylinder, the workload that the benchmark is quoted on, tuned as there
        dict(name="channel_mixed", op="project", geometry="channel", dim=2, n0=1024, n1=512, nodes=400000,
             precision="mixed", tune=True),
        # the same in plain FP64
        dict(name="channel_fp64", op="project", geometry="channel", dim=2, n0=1024, n1=512, nodes=400000,
             precision="fp64", tune=True),
        # one time step's force iteration on the same channel
        dict(name="channel_ib_mixed", op="ib", geometry="channel", dim=2, n0=1024, n1=512, nodes=400000,
             precision="mixed", tol=1e-3),
        # a full time step on the regular (vertex) grid: predictor, direct divergence, DCT-I and
        # quarter-wave passes
        dict(name="vertex_step_mixed", op="step", geometry="channel", dim=2, n0=512, n1=256, nodes=130000,
             precision="mixed", grid="vertices"),
        # a box with a sphere, walls on all sides (zero mode), FP32 velocities
        dict(name="sphere_256x128x128_mixed", op="project", geometry="sphere", dim=3, n0=256, n1=128, n2=128,
             precision="mixed", dtype="f32", tune=True),
        # a 3D request in plain FP64
        dict(name="box_96_fp64", op="project", geometry="box", dim=3, n0=96, n1=96, n2=96, bc="WW,WW,WW",
             precision="fp64", obstacles=1),
        # throughput: uneven 2D problems of the batch workload
        dict(name="batch_64_mixed", op="batch", dim=2, count=64, smallest=64, largest=512, precision="mixed"),
        # requests of the stream that arrived together, 2D and 3D, through the batch executor
        dict(name="serve_12_mixed", op="serve", dim=3, count=12, smallest=128, largest=512, smallest3=64, largest3=96,
             precision="mixed"),
        # the solve alone on a large 3D grid, every axis with walls
        dict(name="poisson_192_mixed", op="poisson", dim=3, n0=192, n1=192, n2=192, bc="WW,WW,WW", precision="mixed"),
    ]


def _lengths(lo, hi):
    """Axis lengths the transforms take: even, half of them 2^a 3^b 5^c."""
    out = []
    for n in range(lo, hi + 1):
        m = n // 2
        for f in (2, 3, 5):
            while m and m % f == 0:
                m //= f
        if n % 2 == 0 and m == 1:
            out.append(n)
    return out


def _length(rng, lo, hi):
    want = math.exp(rng.uniform(math.log(lo), math.log(hi)))
    return min(_lengths(lo, hi), key=lambda n: (abs(n - want), n))


def draw(rng):
    op = rng.choice(["project", "project", "project", "project", "ib", "step", "batch", "serve", "poisson", "poisson"])
    precision = rng.choice(["mixed", "mixed", "fp64", "fp32"])
    bcs = ["PP", "WW", "ID", "DD", "DW"]
    if op == "batch":
        lo = rng.choice([32, 48, 64, 96])
        return dict(op=op, dim=2, count=rng.randint(3, 48), smallest=lo, largest=rng.choice([192, 256, 384, 400]),
                    precision=rng.choice(["mixed", "mixed", "fp32"]))
    if op == "serve":
        return dict(op=op, dim=3, count=rng.randint(2, 12), smallest=_length(rng, 64, 200), largest=_length(rng, 250, 512),
                    smallest3=rng.choice([32, 48, 64]), largest3=rng.choice([72, 80, 96]), precision="mixed")
    if op in ("ib", "step") or (op == "project" and rng.random() < 0.25):
        n1 = _length(rng, 64, 480)
        vertices = op == "step" and rng.random() < 0.5
        case = dict(op=op, geometry="channel", dim=2, n0=2 * n1, n1=n1, nodes=max(130000, int(n1 * n1 * 1.5)),
                    precision=rng.choice(["mixed", "mixed", "fp64"]))
        if op == "ib":
            case["tol"] = rng.choice([1e-2, 1e-3])
        if vertices:
            case["grid"] = "vertices"
        return case
    if op == "poisson":
        dim = rng.choice([2, 3])
        n = [_length(rng, 16, 1024) for _ in range(2)] if dim == 2 else [_length(rng, 16, 160) for _ in range(3)]
        case = dict(op=op, dim=dim, n0=n[0], n1=n[1], bc=",".join(rng.choice(bcs) for _ in range(dim)), precision=precision)
        if dim == 3:
            case["n2"] = n[2]
        if rng.random() < 0.3:
            case["grid"] = "vertices"
        return case
    dim = rng.choice([2, 2, 3])
    n = [_length(rng, 16, 720) for _ in range(2)] if dim == 2 else [_length(rng, 16, 96) for _ in range(3)]
    case = dict(op=op, geometry="box", dim=dim, n0=n[0], n1=n[1], bc=",".join(rng.choice(bcs) for _ in range(dim)),
                precision=precision, dtype=rng.choice(["f64", "f64", "f32"]), obstacles=rng.randint(0, 1),
                force=rng.random() < 0.3)
    if dim == 3:
        case["n2"] = n[2]
    if dim == 2 and rng.random() < 0.2:
        case["knn"] = rng.choice([10, 14, 16])
    if rng.random() < 0.15:
        case["div"] = "wls_direct"
    return case


# ----------------------------------------------------------------------------- inputs

def _shape(case):
    return tuple(case["n%d" % a] for a in range(case["dim"]))


def _pairs(case):
    """Boundary letters at the low and the high end of every axis."""
    bc = case["bc"].split(",")
    return tuple(b[0] for b in bc), tuple(b[1] for b in bc)


def _box(dim, n, lo, hi, obstacles, seed, force=False, dtype="f64", knn=None):
    """Jittered lattice at the grid spacing in a box whose shorter side is 1, with a circle or
    sphere of 10-30% of it."""
    rng = np.random.default_rng(seed)
    h = 1.0 / min(n)
    obs = []
    for _ in range(obstacles):
        d = rng.uniform(0.1, 0.3)
        c = tuple(float(rng.uniform(0.5 * d + 0.1, m * h - 0.5 * d - 0.1)) for m in n)
        obs.append(("circle" if dim == 2 else "sphere", c, 0.5 * d))
    return wl.generic(dim=dim, n=n, h=(h,) * dim, bc_lo=lo, bc_hi=hi, obstacles=obs, seed=int(rng.integers(1 << 31)),
                      with_force=force, knn=knn, dtype=np.float32 if dtype == "f32" else np.float64)


_clouds = {}


def _geometries(case):
    """The problem, or the problems of a batch, of a case: the nodes do not depend on the seed, as
    a program keeps its nodes while the velocity changes. The last few are kept."""
    key = repr(sorted((k, v) for k, v in case.items() if k not in ("name", "op", "precision", "tol", "tune", "grid", "div")))
    key = (case["op"] if case["op"] in ("batch", "serve") else "one", key)
    if key not in _clouds:
        while len(_clouds) >= 8:
            del _clouds[next(iter(_clouds))]
        _clouds[key] = _draw_geometries(case, 14690)
    return _clouds[key]


def _draw_geometries(case, seed):
    if case["op"] == "batch":
        sizes = [n for n in wl.BATCH_SIZES + (32, 48, 100, 160, 240, 320, 400) if case["smallest"] <= n <= case["largest"]]
        if case["smallest"] == 64 and case["largest"] == 512:
            sizes = list(wl.BATCH_SIZES)
        return wl.batch_2d(count=case["count"], seed=seed, sizes=sizes)
    if case["op"] == "serve":
        two = [n for n in (64, 100, 128, 192, 200, 256, 384, 400, 512) if case["smallest"] <= n <= case["largest"]]
        three = [n for n in (32, 48, 64, 72, 80, 96) if case["smallest3"] <= n <= case["largest3"]]
        rng = np.random.default_rng(seed)
        out = []
        for i in range(case["count"]):     # seven of ten requests are 2D
            if i % 10 < 7:
                out.append(_box(2, (int(rng.choice(two)),) * 2, ("I", "W"), ("D", "W"), 1, int(rng.integers(1 << 31))))
            else:
                out.append(_box(3, (int(rng.choice(three)),) * 3, ("W",) * 3, ("W",) * 3, 1, int(rng.integers(1 << 31))))
        return out
    if case["geometry"] == "taylor_green":
        return [wl.periodic_taylor_green(n=case["n0"], seed=seed)]
    if case["geometry"] == "channel":
        return [wl.channel_cylinder(case["n0"], case["n1"], case["nodes"], seed)]
    if case["geometry"] == "sphere":
        return [wl.box_sphere(_shape(case), seed)]
    lo, hi = _pairs(case)
    return [_box(case["dim"], _shape(case), lo, hi, case["obstacles"], seed, case.get("force", False),
                 case.get("dtype", "f64"), case.get("knn"))]


def _problems(case, seed):
    """The case's problems with the velocities of the seed: the geometry's field scaled (as the
    request stream scales it) plus a few smooth modes, zero at virtual nodes."""
    rng = np.random.default_rng(seed)
    out = []
    for q in _geometries(case):
        x = torch.as_tensor(q.nodes, device=_dev())
        u = float(rng.uniform(0.5, 1.5)) * torch.as_tensor(q.u_star, device=x.device).double()
        for _ in range(4):
            k = [2.0 * math.pi * int(rng.integers(1, 9)) / length for length in q.lengths()]
            wave = torch.ones_like(x[0])
            for a in range(q.dim):
                wave = wave * torch.cos(k[a] * (x[a] - q.lo[a]))
            u += 0.1 * torch.as_tensor(rng.normal(size=(q.dim, 1)), device=x.device) * wave
        u[:, torch.as_tensor(q.node_type == wl.VIRTUAL, device=x.device)] = 0.0
        f = None if q.f_ib is None else float(rng.uniform(0.5, 1.5)) * q.f_ib
        out.append(dataclasses.replace(q, u_star=u.cpu().numpy().astype(q.u_star.dtype), f_ib=f))
    return out


def _source(case, seed):
    """Source of the solve alone: a smooth field and noise, on the unknowns of the grid."""
    shape = _unknowns(case)
    g = torch.Generator(device="cuda").manual_seed(seed)
    s = 0.1 * torch.randn(shape, generator=g, device="cuda", dtype=torch.float64)
    k = torch.randint(1, 6, (6, case["dim"]), generator=g, device="cuda").tolist()
    for m in k:
        term = torch.ones((), device="cuda", dtype=torch.float64)
        for a, n in enumerate(shape):
            x = (torch.arange(n, device="cuda", dtype=torch.float64) + 0.5) / n
            term = term * torch.cos(math.pi * m[a] * x).reshape([-1 if b == a else 1 for b in range(case["dim"])])
        s = s + term
    return s.contiguous()


def _unknowns(case):
    if case.get("grid", "cells") == "cells":
        return _shape(case)
    lo, hi = _pairs(case)
    return tuple(pc.vertex_unknowns(lo[a], hi[a], n) for a, n in enumerate(_shape(case)))


def _spacing(case):
    return (1.0 / min(_shape(case)),) * case["dim"]


def _dt(problem):
    """A step at a CFL number of about 0.2."""
    return 0.2 * min(problem.h) / max(1.0, float(np.abs(problem.u_star).max()))


def prepare(case, seed):
    if case["op"] == "poisson":
        lo, hi = _pairs(case)
        plan = pc.GridPlan(case["dim"], _shape(case), _spacing(case), lo, hi, precision=case["precision"],
                           grid_type=case.get("grid", "cells"))
        s = _source(case, seed)
        return dict(op="poisson", plan=plan, s=s, p=torch.empty_like(s))
    problems = _problems(case, seed)
    options = dict(precision=case["precision"])
    if case.get("grid", "cells") == "vertices":
        options.update(grid_type="vertices", div_mode="wls_direct")
    elif case.get("div"):
        options.update(div_mode=case["div"])
    plans = [pc.Plan(q, **options) for q in problems]
    u = [torch.as_tensor(q.u_star, device="cuda") for q in problems]
    if case["op"] in ("batch", "serve"):
        # one array per kind of output, each problem a view of it
        whole = [torch.empty(sum(math.prod(p.shape) for p in plans), dtype=torch.float64, device="cuda")]
        whole += [torch.empty(sum(v.numel() for v in u), dtype=torch.float64, device="cuda") for _ in range(2)]
        at = [0, 0]
        args = []
        for q, plan, v in zip(problems, plans, u):
            np_, nv = math.prod(plan.shape), v.numel()
            args.append(dict(dt=q.dt, u_star=v, f_ib=None, p=whole[0][at[0]:at[0] + np_].view(plan.shape),
                             u=whole[1][at[1]:at[1] + nv].view(v.shape), f=whole[2][at[1]:at[1] + nv].view(v.shape)))
            at = [at[0] + np_, at[1] + nv]
        state = dict(op=case["op"], plans=plans, args=args, out=dict(p=whole[0], u=whole[1], f=whole[2]))
        if case["op"] == "serve":
            state["batcher"] = pc.Batcher()
        return state
    plan, problem = plans[0], problems[0]
    if case.get("tune"):
        plan.autotune()
    state = dict(op=case["op"], plan=plan, u=u[0], f_ib=None, dt=problem.dt, out=plan.alloc_outputs(),
                 tol=case.get("tol"))
    if problem.f_ib is not None:
        state["f_ib"] = torch.as_tensor(problem.f_ib, device="cuda")
    if case["op"] == "step":
        state["dt"] = _dt(problem)
        state["momentum"] = pc.Momentum(plan, nu=1e-3)
        state["u_star"] = torch.empty_like(u[0])
        # the flow has been running: the step before this one left its right-hand side
        state["momentum"].predict(0.98 * u[0], state["dt"], out=state["u_star"])
    return state


def run(state):
    op = state["op"]
    if op == "poisson":
        return state["plan"].solve_poisson(state["s"], p_out=state["p"])[0]
    if op == "batch":
        pc.project_batch(state["plans"], state["args"])
        return state["out"]
    if op == "serve":
        state["batcher"].launch(state["plans"], state["args"])
        return state["out"]
    if op == "ib":
        p, u, f, info = state["plan"].project_ib(state["u"], tol=state["tol"], dt=state["dt"], out=state["out"])
        return dict(p=p, u=u, f=f, iterations=info["iterations"])
    if op == "step":
        u_star = state["momentum"].predict(state["u"], state["dt"], out=state["u_star"])
        p, u, f, _ = state["plan"].project(u_star, dt=state["dt"], out=state["out"])
        return dict(u_star=u_star, p=p, u=u, f=f)
    p, u, f, _ = state["plan"].project(state["u"], f_ib=state["f_ib"], dt=state["dt"], out=state["out"])
    return dict(p=p, u=u, f=f)


# ----------------------------------------------------------------------------- work

def _solve_work(shape):
    cells = math.prod(shape)
    return 2 * 2.5 * cells * sum(math.log2(n) for n in shape) + cells


def _project_work(shape, nodes, vb, knn=None, force=False, direct=False):
    """WLS rows (4-byte columns, 8-byte weights) and node values read once, results written once."""
    dim, cells = len(shape), math.prod(shape)
    k, kg = knn or (12 if dim == 2 else 27), 3 ** dim
    rows = cells * k * (4 + 8 * dim) if direct else dim * cells * k * 12
    data = rows + nodes * kg * (4 + 8 * dim) + nodes * (1 + dim * vb * (4 if force else 3)) + 8 * cells
    return data, 2 * dim * k * cells + 2 * dim * kg * nodes + _solve_work(shape)


def work(case):
    if case["op"] == "poisson":
        shape = _unknowns(case)
        return dict(bytes=16 * math.prod(shape), flops=_solve_work(shape))
    if case["op"] in ("batch", "serve"):
        total = [0, 0]
        for i in range(case["count"]):
            if case["op"] == "serve" and i % 10 >= 7:
                shape = (0.5 * (case["smallest3"] + case["largest3"]),) * 3
            else:
                shape = (0.5 * (case["smallest"] + case["largest"]),) * 2
            b, f = _project_work(shape, math.prod(shape), 8)
            total = [total[0] + b, total[1] + f]
        return dict(bytes=total[0], flops=total[1])
    shape = _shape(case)
    nodes = case.get("nodes", math.prod(shape))
    vb = 4 if case.get("dtype") == "f32" or case["geometry"] == "sphere" else 8
    b, f = _project_work(shape, nodes, vb, case.get("knn"), case.get("force", False),
                         case.get("div") == "wls_direct" or case.get("grid") == "vertices")
    if case["op"] == "step":
        b += nodes * (12 * (4 + 8 * 3) + 6 * 2 * 8)
        f += nodes * 2 * 12 * 3 * 2
    if case["op"] == "ib":       # at least one more solve and the force at the boundary nodes
        f += _solve_work(shape)
    return dict(bytes=b, flops=f)


# ----------------------------------------------------------------------------- 64-bit values
# The method in plain torch: nearest nodes, weighted least squares by batched LU, dense eigenbases.

def _dev():
    return torch.device("cuda" if torch.cuda.is_available() else "cpu")


def _min_image(delta, lengths, periodic):
    for a, per in enumerate(periodic):
        if per:
            delta[..., a] -= lengths[a] * torch.round(delta[..., a] / lengths[a])
    return delta


def _nearest(points, queries, k, lo, lengths, periodic):
    """Indices (Q, k) of the k nearest points: a bucket table searched in growing windows."""
    dim, dev = points.shape[1], points.device
    n = points.shape[0]
    cell = (2.0 * math.prod(lengths) / n) ** (1.0 / dim)
    nb = [max(1, int(v / cell)) for v in lengths]
    size = torch.tensor([lengths[a] / nb[a] for a in range(dim)], device=dev, dtype=torch.float64)
    low = torch.tensor(lo, device=dev, dtype=torch.float64)
    top = torch.tensor(nb, device=dev) - 1
    bucket = lambda x: torch.minimum(((x - low) / size).floor().long().clamp(min=0), top)  # noqa: E731

    def flat(b):
        f = b[..., 0]
        for a in range(1, dim):
            f = f * nb[a] + b[..., a]
        return f

    pid = flat(bucket(points))
    order = torch.argsort(pid, stable=True)
    count = torch.bincount(pid, minlength=math.prod(nb))
    start = torch.cumsum(count, 0) - count
    most = int(count.max())
    table = torch.full((math.prod(nb) + 1, most), -1, device=dev, dtype=torch.int32)
    table[pid[order], torch.arange(n, device=dev) - start[pid[order]]] = order.int()
    out = torch.empty((queries.shape[0], k), device=dev, dtype=torch.long)
    todo, ring = torch.arange(queries.shape[0], device=dev), 2
    while todo.numel():
        whole = any(2 * ring + 1 > nb[a] for a in range(dim))     # the window is the whole box
        if whole:
            width = n
        else:
            span = torch.arange(-ring, ring + 1, device=dev)
            offs = torch.stack(torch.meshgrid(*[span] * dim, indexing="ij"), -1).reshape(-1, dim)
            width = offs.shape[0] * most
        left = []
        for part in torch.split(todo, max(1, 60_000_000 // width)):
            q = queries[part]
            if whole:
                cand = torch.arange(n, device=dev, dtype=torch.int32).expand(part.numel(), n)
            else:
                b = bucket(q)[:, None, :] + offs
                ok = torch.ones(b.shape[:-1], device=dev, dtype=torch.bool)
                for a in range(dim):
                    if periodic[a]:
                        b[..., a] %= nb[a]
                    else:
                        ok &= (b[..., a] >= 0) & (b[..., a] < nb[a])
                cand = table[torch.where(ok, flat(b), table.shape[0] - 1)].reshape(part.numel(), -1)
            j = cand.long().clamp(min=0)
            d2 = torch.zeros(cand.shape, device=dev, dtype=torch.float64)
            for a in range(dim):
                x = points[:, a][j] - q[:, a, None]
                if periodic[a]:
                    x = x - lengths[a] * torch.round(x / lengths[a])
                d2 += x * x
            d2[cand < 0] = math.inf
            d2, sel = torch.topk(d2, k, dim=1, largest=False)
            done = torch.full_like(part, whole, dtype=torch.bool) | (d2.amax(1) < (ring * float(size.min())) ** 2)
            out[part[done]] = torch.gather(j, 1, sel)[done]
            left.append(part[~done])
        todo, ring = torch.cat(left), ring + 2
    return out


def _rows(points, queries, idx, lengths, periodic, want):
    """Least-squares rows of the quadratic basis: value (Q, k), gradient (dim, Q, k) or gradient
    and Laplacian (dim + 1, Q, k)."""
    k, dim = idx.shape[1], points.shape[1]
    out = []
    for at in torch.split(torch.arange(queries.shape[0], device=points.device), 200_000):
        delta = _min_image(points[idx[at]] - queries[at][:, None, :], lengths, periodic)
        d2 = (delta * delta).sum(-1)
        c = math.sqrt(math.pi / k) if dim == 2 else (4.0 * math.pi / (3.0 * k)) ** (1.0 / 3.0)
        hs = SUPPORT * c * d2.amax(1).sqrt()
        w = torch.where(d2 <= hs[:, None] ** 2, torch.exp(-EPS * d2 / hs[:, None] ** 2), torch.zeros_like(d2))
        x = delta / hs[:, None, None]
        q = [torch.ones_like(d2)] + [x[..., a] for a in range(dim)]
        second = []
        for a in range(dim):
            for b in range(a, dim):
                if a == b:
                    second.append(len(q))
                q.append((0.5 if a == b else 1.0) * x[..., a] * x[..., b])
        q = torch.stack(q, -1)
        wq = w[..., None] * q
        rhs = torch.zeros((at.numel(), q.shape[-1], 1 if want == "value" else dim + (want == "laplacian")),
                          device=points.device, dtype=torch.float64)
        if want == "value":
            rhs[:, 0, 0] = 1.0
        else:
            for a in range(dim):
                rhs[:, 1 + a, a] = 1.0 / hs
            if want == "laplacian":
                for m in second:
                    rhs[:, m, dim] = 1.0 / hs ** 2
        y = torch.linalg.solve(wq.transpose(1, 2) @ q, rhs)
        out.append((wq @ y).permute(2, 0, 1))
    out = torch.cat(out, 1)
    return out[0] if want == "value" else out


def _basis(lo, hi, n, h, vertices, dev):
    """Eigenvectors (columns) and eigenvalues of the 3-point operator of one axis."""
    neu = lambda c: c in "WI"  # noqa: E731
    kind = "P" if lo == "P" else ("N" if neu(lo) else "D") + ("N" if neu(hi) else "D")
    if vertices and kind != "P":
        j = torch.arange({"NN": n + 1, "DD": n - 1}.get(kind, n), device=dev, dtype=torch.float64) + (kind[0] == "D")
    else:
        j = torch.arange(n, device=dev, dtype=torch.float64) + (0.0 if vertices else 0.5)
    k = torch.arange(j.numel(), device=dev, dtype=torch.float64)
    if kind == "P":
        j = torch.arange(n, device=dev, dtype=torch.float64)
        w = torch.ceil(k / 2)
        theta = 2.0 * math.pi * w / n
        phase = torch.remainder(w[None, :] * j[:, None], n) * (2.0 * math.pi / n)
        phi = torch.where((k[None, :] % 2 == 1) | (k[None, :] == 0), torch.cos(phase), torch.sin(phase))
    else:
        theta = math.pi * (k + {"NN": 0.0, "DD": 1.0}.get(kind, 0.5)) / n
        phi = (torch.cos if kind[0] == "N" else torch.sin)(theta[None, :] * j[:, None])
    return phi, -(4.0 / (h * h)) * torch.sin(theta / 2.0) ** 2, kind


def _poisson(s, lo, hi, n, h, vertices=False):
    """p with L_h p = s (the constant dropped where no end is Dirichlet)."""
    dim = s.dim()
    basis = [_basis(lo[a], hi[a], n[a], h[a], vertices, s.device) for a in range(dim)]
    apply = lambda m, x, a: torch.movedim(torch.tensordot(m, x, dims=([1], [a])), 0, a)  # noqa: E731
    c = s
    for a in range(dim):
        phi = basis[a][0]
        if vertices:
            xa = torch.movedim(c, a, 0)
            c = torch.movedim(torch.linalg.solve(phi, xa.reshape(xa.shape[0], -1)).reshape(xa.shape), 0, a)
        else:
            c = apply((phi / (phi * phi).sum(0)).T, c, a)
    lam = 0.0
    for a in range(dim):
        lam = lam + basis[a][1].reshape([-1 if b == a else 1 for b in range(dim)])
    if all(b[2] in ("P", "NN") for b in basis):
        first = (0,) * dim
        c = c.clone()
        c[first] = 0.0
        lam[first] = 1.0
    c = c / lam
    for a in range(dim):
        c = apply(basis[a][0], c, a)
    return c


class _Exact:
    """One problem's rows, and a pass of the pressure correction on them."""

    def __init__(self, q, vertices=False, direct=False):
        dev = _dev()
        self.q, self.vertices, self.direct = q, vertices, direct or vertices
        self.lengths = q.lengths()
        self.periodic = [b == "P" for b in q.bc_lo]
        self.pts = torch.as_tensor(q.nodes, device=dev).T.contiguous()
        self.ib = torch.as_tensor(q.node_type, device=dev) != wl.FLUID
        d = q.dim
        grid = lambda axes: torch.stack(torch.meshgrid(*axes, indexing="ij"), -1).reshape(-1, d)  # noqa: E731
        centre = [q.lo[a] + (torch.arange(q.n[a], device=dev, dtype=torch.float64) + 0.5) * q.h[a] for a in range(d)]
        vertex = [q.lo[a] + torch.arange(q.n[a] + (not self.periodic[a]), device=dev, dtype=torch.float64) * q.h[a]
                  for a in range(d)]
        self.rows = []
        if self.direct:
            axes = centre
            if vertices:        # the unknowns: Dirichlet ends left out
                self.cut = [slice(int(q.bc_lo[a] == "D"), vertex[a].numel() - int(q.bc_hi[a] == "D")) for a in range(d)]
                axes = [vertex[a][self.cut[a]] for a in range(d)]
            self.shape = tuple(x.numel() for x in axes)
            at = grid(axes)
            idx = _nearest(self.pts, at, q.knn, q.lo[:d], self.lengths, self.periodic)
            self.rows = [(idx, _rows(self.pts, at, idx, self.lengths, self.periodic, "gradient"))]
        else:
            self.shape = tuple(q.n[:d])
            for a in range(d):
                at = grid([vertex[b] if b == a else centre[b] for b in range(d)])
                idx = _nearest(self.pts, at, q.knn, q.lo[:d], self.lengths, self.periodic)
                w = _rows(self.pts, at, idx, self.lengths, self.periodic, "value")
                w = w.reshape(tuple((vertex if b == a else centre)[b].numel() for b in range(d)) + (q.knn,)).clone()
                if q.bc_lo[a] == "W":
                    w.select(a, 0).zero_()
                if q.bc_hi[a] == "W":
                    w.select(a, w.shape[a] - 1).zero_()
                self.rows.append((idx.reshape(w.shape), w))
        # the block of 3^d pressure points around each node
        block = torch.zeros((self.pts.shape[0], 1), device=dev, dtype=torch.long)
        lattice = vertex if vertices else centre
        self.full = tuple(x.numel() for x in lattice)
        for a in range(d):
            m = self.full[a]
            x = (self.pts[:, a] - q.lo[a]) / q.h[a] + (0.5 if vertices else 0.0)
            c = x.floor().long()
            if vertices and self.periodic[a]:
                c = c % m
            b = c.clamp(0, m - 1)[:, None] - 1
            b = b + torch.arange(3, device=dev) if self.periodic[a] else b.clamp(0, m - 3) + torch.arange(3, device=dev)
            block = (block[:, :, None] * m + (b % m)[:, None, :]).reshape(self.pts.shape[0], -1)
        self.block = block
        self.grad = _rows(grid(lattice), self.pts, block, self.lengths, self.periodic, "gradient")

    def source(self, ut, dt):
        q, d = self.q, self.q.dim
        if self.direct:
            idx, g = self.rows[0]
            return sum((g[a] * ut[a][idx]).sum(-1) for a in range(d)).reshape(self.shape) / (BETA * dt)
        s = 0.0
        for a in range(d):
            flux = (self.rows[a][1] * ut[a][self.rows[a][0]]).sum(-1)
            if self.periodic[a]:
                flux = torch.cat([flux, flux.narrow(a, 0, 1)], a)
            s = s + torch.diff(flux, dim=a) / q.h[a]
        return s / (BETA * dt)

    def project(self, u, f, dt):
        q, d = self.q, self.q.dim
        s = self.source(u if f is None else u + dt * f, dt)
        p = _poisson(s, q.bc_lo, q.bc_hi, q.n, q.h, self.vertices)
        field = p
        if self.vertices:
            field = torch.zeros(self.full, device=p.device, dtype=p.dtype)
            field[tuple(self.cut)] = p
        v = field.reshape(-1)[self.block]
        g = torch.stack([(self.grad[a] * v).sum(-1) for a in range(d)])
        un = torch.where(self.ib, torch.zeros_like(u), u - BETA * dt * g)
        fn = torch.where(self.ib, -u / dt + BETA * g, torch.zeros_like(u))
        return p, un, fn


def exact(case, seed):
    if case["op"] == "poisson":
        lo, hi = _pairs(case)
        return _poisson(_source(case, seed), lo, hi, _shape(case), _spacing(case), case.get("grid", "cells") == "vertices")
    if case.get("geometry") == "sphere":
        return None         # twelve million least-squares rows
    problems = _problems(case, seed)
    dev = _dev()
    vertices = case.get("grid", "cells") == "vertices"
    all_p, all_u, all_f = [], [], []
    for q in problems:
        e = _Exact(q, vertices, case.get("div") == "wls_direct")
        u = torch.as_tensor(q.u_star, device=dev).double()
        f = None if q.f_ib is None else torch.as_tensor(q.f_ib, device=dev).double()
        if case["op"] == "step":
            dt = _dt(q)
            idx = _nearest(e.pts, e.pts, q.knn, q.lo[:q.dim], e.lengths, e.periodic)
            rows = _rows(e.pts, e.pts, idx, e.lengths, e.periodic, "laplacian")
            kind = torch.as_tensor(q.node_type, device=dev)

            def rhs(v):
                d = torch.stack([(rows[r] * v[:, idx]).sum(-1) for r in range(q.dim + 1)])
                return 1e-3 * d[q.dim] - sum(v[b] * d[b] for b in range(q.dim))

            before = 0.98 * u
            r0 = rhs(before)
            star0 = torch.where(kind == wl.FLUID, before + dt * r0, torch.zeros_like(u))
            gp = (star0 - u) / (BETA * dt)
            star = torch.where(kind == wl.FLUID, u + dt * (1.5 * rhs(u) - 0.5 * (r0 - gp)), torch.zeros_like(u))
            p, un, fn = e.project(star, None, dt)
            return dict(u_star=star, p=p, u=un, f=fn)
        if case["op"] == "ib":
            f = torch.zeros_like(u)
            for it in range(1, 51):
                p, un, fn = e.project(u, f, q.dt)
                diff = float(((fn - f)[:, e.ib] ** 2).sum())
                prev = float((f[:, e.ib] ** 2).sum())
                f = fn
                if diff <= case["tol"] * prev if prev else diff == 0.0:
                    break
            return dict(p=p, u=un, f=fn, iterations=it)
        p, un, fn = e.project(u, f, q.dt)
        if case["op"] == "project":
            return dict(p=p, u=un, f=fn)
        all_p.append(p.reshape(-1))
        all_u.append(un.reshape(-1))
        all_f.append(fn.reshape(-1))
    return dict(p=torch.cat(all_p), u=torch.cat(all_u), f=torch.cat(all_f))
