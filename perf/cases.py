"""Timed work of the library, through its public entry points.

Every case is one call, or one short sequence of calls, that a program using
the library makes: clouds of 1,000 to 500,000 oriented points on grids of 24^3
to 512^3, forward alone and with the adjoint, interpolated and exact queries,
and normals estimated from raw points.  ``kind`` names the sequence:

  forward      reconstruct: signed distance grid and unit normals
  moving       four reconstructions of a body that moves, on a warm-start handle
  step         reconstruct, interpolate phi at query points, adjoint of the query
  grid_step    sdf_grid and its backward from seeds on the whole grid
  shape        spherical-harmonic parameters -> points -> phi at queries -> d/dtheta
  query        phi and normals interpolated at query points of a kept forward
  query_exact  exact off-grid distances and their gradients on a kept forward
  exact_step   sdf_query_exact and its backward
  normals      raw points -> D-PCA normals -> parity orientation

``exact`` restates each of them in 64-bit torch (dense cosine transforms, a
brute-force nearest triangle behind a conservative cull, gradients by autograd).
"""
from __future__ import annotations

import functools
import math

import numpy as np
import torch

import paper_2609_20964_gb300 as wgeo

BBOX = np.array([0, 0, 0, 1, 1, 1], dtype=np.float32)
CENTRE = 0.5
WAVE_STEPS = 4
F64 = torch.float64


# ---------------------------------------------------------------- the cases
def listed():
    base = dict(body="star", precision="mixed", galerkin=0)
    return [
        # the smallest grid and cloud in use (a sphere, 4,096 points): latency and launches
        dict(base, name="forward_64", kind="forward", body="sphere", res=64, n=4096),
        # the commonest request of the serving mix, with gradients
        dict(base, name="step_64", kind="step", res=64, n=16_384, m=50_000),
        # exact queries differentiated on a ragged grid (multigrid solver), odd counts
        dict(base, name="exact_step_88", kind="exact_step", res=88, n=30_011, m=101_003),
        # the unlumped Galerkin operator, forward and adjoint
        dict(base, name="step_galerkin_96", kind="step", res=96, n=40_000, m=100_000, galerkin=1),
        # a loss on the whole grid, ragged grid (multigrid solver in both directions)
        dict(base, name="grid_step_120", kind="grid_step", res=120, n=60_000),
        # the differentiable shape workload: 49 parameters, 100,000 points, 500,000 queries
        dict(base, name="shape_128", kind="shape", res=128, n=100_000, m=500_000, lmax=6),
        # interpolation alone, as after a forward whose grid serves many query batches
        dict(base, name="query_128", kind="query", res=128, n=100_000, m=1_000_000),
        # the moving-boundary workload: the swimming ellipsoid, each step warm-started
        dict(base, name="moving_192", kind="moving", body="wave", res=192, n=50_000),
        # the benchmark step: noisy star body, forward + query + adjoint
        dict(base, name="step_256", kind="step", res=256, n=200_000, m=1_000_000, noise=0.002),
        # exact distances at a million points
        dict(base, name="query_exact_256", kind="query_exact", res=256, n=200_000, m=1_000_000, noise=0.002),
        # raw points to oriented normals on the benchmark cloud's size
        dict(base, name="normals_200k", kind="normals", n=200_000, radius=0.1),
        # the largest grid of the direct solver and the largest cloud
        dict(base, name="forward_512", kind="forward", res=512, n=500_000, noise=0.001),
    ]


def _log_uniform(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def _grid(rng, lo, hi):
    """A grid size the library takes (m * 2^k, m <= 16), log-uniform in [lo, hi]."""
    r = _log_uniform(rng, lo, hi)
    step = 1
    while 16 * step < r:
        step *= 2
    return max(lo, min(hi, step * int(round(r / step))))


def draw(rng):
    kind = rng.choice(["forward", "forward", "step", "step", "grid_step", "exact_step", "shape", "query",
                       "query_exact", "moving", "normals"])
    if kind == "normals":
        n = int(_log_uniform(rng, 10_000, 200_000))
        return dict(kind=kind, body="star", precision="mixed", galerkin=0, n=n, radius=round(rng.uniform(0.06, 0.1), 4))
    res = _grid(rng, 24, 256)
    n = int(_log_uniform(rng, max(1000, res * res // 3), 500_000 if res > 64 else 100_000))
    case = dict(kind=kind, body=rng.choice(["sphere", "star", "star"]), precision="mixed", galerkin=0, res=res, n=n)
    if kind == "moving":
        case["body"] = "wave"
    if kind == "shape":
        case.update(body="star", lmax=rng.randint(3, 8))
    if kind == "forward" and rng.random() < 0.3:
        case["precision"] = "fp32"
    elif kind == "step" and rng.random() < 0.3:
        case["galerkin"] = 1
    if kind not in ("forward", "moving", "grid_step"):
        case["m"] = int(_log_uniform(rng, 1000, 1_000_000))
    return case


# ---------------------------------------------------------------- inputs
def _generator(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(int(seed))
    return g


def _directions(k, g):
    u = torch.randn(k, 3, generator=g, device="cuda", dtype=F64)
    return u / u.norm(dim=1, keepdim=True)


def _weighted(u, weight, n, g):
    """n of the directions u, drawn without replacement in proportion to weight."""
    key = -torch.log(torch.rand(len(u), generator=g, device="cuda", dtype=F64)) / weight
    return u[torch.topk(key, n, largest=False).indices]


def _legendre(l, t):
    """P_l(t) and its derivative, each row of t with its own degree l (2..8)."""
    p0, p1 = torch.ones_like(t), t
    d0, d1 = torch.zeros_like(t), torch.ones_like(t)
    p, d = p1, d1
    for k in range(2, 9):
        p0, p1 = p1, ((2 * k - 1) * t * p1 - (k - 1) * p0) / k
        d0, d1 = d1, d0 + (2 * k - 1) * p0
        p, d = torch.where(l == k, p1, p), torch.where(l == k, d1, d)
    return p, d


def _star(n, noise, g):
    """A star body r(u) = 0.3 + a sum of 24 zonal harmonics of degree 2 to 8
    about random axes, within [0.16, 0.44]; area-uniform samples, analytic
    normals, then Gaussian position noise."""
    axes = _directions(24, g)
    l = torch.randint(2, 9, (24, 1), generator=g, device="cuda")
    a = torch.randn(24, 1, generator=g, device="cuda", dtype=F64) * 0.02

    def radius(u):
        p, d = _legendre(l, axes @ u.T)
        grad = ((a * d).T @ axes)
        return (a * p).sum(0), grad - (grad * u).sum(1, keepdim=True) * u

    u = _directions(4 * n + 4096, g)
    r, grad = radius(u)
    scale = min(1.0, 0.14 / float(r.abs().max()))
    r = 0.3 + scale * r
    u = _weighted(u, r * torch.sqrt(r * r + scale * scale * (grad * grad).sum(1)), n, g)
    r, grad = radius(u)
    r = (0.3 + scale * r)[:, None]
    nrm = u - scale * grad / r
    pts = CENTRE + r * u + noise * torch.randn(n, 3, generator=g, device="cuda", dtype=F64)
    return pts.float(), (nrm / nrm.norm(dim=1, keepdim=True)).float()


def _wave(n, t, g, axes=(0.35, 0.08, 0.12), amp=0.04, length=0.9, period=200):
    """An ellipsoid bent by a lateral travelling wave at step t."""
    ax = torch.tensor(axes, device="cuda", dtype=F64)
    u = _directions(8 * n, g)
    u = _weighted(u, (u / ax).norm(dim=1), n, g)
    p, nrm = CENTRE + u * ax, u / ax
    s = (p[:, 0] - (CENTRE - axes[0])) / (2 * axes[0])
    ph = 2 * math.pi * (s / length - t / period)
    slope = (2 * amp * s * torch.sin(ph) + amp * s * s * torch.cos(ph) * 2 * math.pi / length) / (2 * axes[0])
    p = torch.stack([p[:, 0], p[:, 1] + amp * s * s * torch.sin(ph), p[:, 2]], 1)
    nrm = torch.stack([nrm[:, 0] - slope * nrm[:, 1], nrm[:, 1], nrm[:, 2]], 1)
    return p.float(), (nrm / nrm.norm(dim=1, keepdim=True)).float()


def _cloud(case, g, t=0):
    if case["body"] == "sphere":
        u = _directions(case["n"], g)
        return (CENTRE + 0.3 * u).float(), u.float()
    if case["body"] == "wave":
        return _wave(case["n"], t, g)
    return _star(case["n"], case.get("noise", 0.0), g)


def _inputs(case, seed):
    g = _generator(seed)
    kind, m = case["kind"], case.get("m", 0)
    x = {}
    if kind == "shape":
        K = (case["lmax"] + 1) ** 2
        x["theta"] = 0.012 * torch.randn(K, generator=g, device="cuda")
        x["dirs"] = _directions(case["n"], g).float()
    elif kind == "moving":
        t0 = int(torch.randint(0, 196, (1,), generator=g, device="cuda"))
        x["clouds"] = [_cloud(case, g, t0 + k) for k in range(WAVE_STEPS)]
    else:
        x["points"], x["normals"] = _cloud(case, g)
    if m:
        x["q"] = torch.rand(m, 3, generator=g, device="cuda")
    if kind in ("step", "exact_step"):
        x["seed_q"] = torch.randn(m, generator=g, device="cuda")
    if kind == "grid_step":
        x["seed_grid"] = torch.randn(case["res"], case["res"], case["res"], generator=g, device="cuda")
    return x


def prepare(case, seed):
    x = _inputs(case, seed)
    kind, n = case["kind"], case["n"]
    options = dict(precision=wgeo.PREC_FP32 if case["precision"] == "fp32" else wgeo.PREC_MIXED,
                   galerkin=case["galerkin"])
    if kind == "moving":
        options["warm_start"] = 1
    res = case.get("res", 16)
    rec = wgeo.Reconstructor(res, n, **options)
    state = dict(case=case, rec=rec, **x)
    if kind in ("query", "query_exact"):
        rec.reconstruct(x["points"], x["normals"], BBOX, res, with_sdf=False, with_normals=False)
    return state


def run(state):
    case, rec = state["case"], state["rec"]
    kind, res = case["kind"], case.get("res")
    if kind == "forward":
        return rec.reconstruct(state["points"], state["normals"], BBOX, res)
    if kind == "moving":
        return [rec.reconstruct(p, nrm, BBOX, res) for p, nrm in state["clouds"]]
    if kind == "step":
        sdf, nrm = rec.reconstruct(state["points"], state["normals"], BBOX, res)
        sdf_q, _ = rec.query(state["q"], with_normals=False)
        dp, dn, _ = rec.backward(q=state["q"], d_sdf_q=state["seed_q"])
        return sdf, nrm, sdf_q, dp, dn
    if kind == "grid_step":
        p, nrm = state["points"].requires_grad_(), state["normals"].requires_grad_()
        sdf, unit = wgeo.sdf_grid(p, nrm, rec, BBOX, res)
        dp, dn = torch.autograd.grad(sdf, (p, nrm), state["seed_grid"])
        return sdf.detach(), unit.detach(), dp, dn
    if kind == "shape":
        theta = state["theta"].requires_grad_()
        p, nrm = wgeo.sh_points(theta, state["dirs"], rec)
        phi, unit = wgeo.sdf_query(p, nrm, state["q"], rec, BBOX, res)
        loss = ((phi - ((state["q"] - CENTRE).norm(dim=1) - 0.3)) ** 2).mean()
        (dtheta,) = torch.autograd.grad(loss, theta)
        return phi.detach(), unit.detach(), dtheta
    if kind == "query":
        return rec.query(state["q"])
    if kind == "query_exact":
        return rec.query_exact(state["q"])
    if kind == "exact_step":
        x = [state[k].requires_grad_() for k in ("points", "normals", "q")]
        phi = wgeo.sdf_query_exact(*x, rec, BBOX, res)
        return (phi.detach(), *torch.autograd.grad(phi, x, state["seed_q"]))
    normals, _ = rec.estimate_normals(state["points"], BBOX, case["radius"])
    rec.orient_normals(state["points"], normals, BBOX)
    return normals


def work(case):
    """Bytes: each input read once, each output written once (and, on a kept
    forward, the grid values read once).  Operations: 40 per point-triangle
    test with one test per node or exact query, the two cosine transforms of a
    direct solve per linear solve, 27 cells of 8 operations per point and pass,
    33 per (point, neighbour) pair of the normal estimation."""
    kind, n, m = case["kind"], case["n"], case.get("m", 0)
    if kind == "normals":
        area = 4 * math.pi * 0.3 ** 2
        pairs = n * max(1.0, n * math.pi * case["radius"] ** 2 / area)
        return {"bytes": 24.0 * n, "flops": 33.0 * pairs}
    cells = float(case["res"]) ** 3
    solve = 2 * 3 * 2.5 * math.log2(case["res"]) * cells
    forward = {"bytes": 24.0 * n + 16.0 * cells, "flops": 40.0 * cells + solve + 27.0 * 8 * n}
    if kind == "forward":
        return forward
    if kind == "moving":
        return {k: WAVE_STEPS * v for k, v in forward.items()}
    if kind == "query":
        return {"bytes": 28.0 * m + 4.0 * cells, "flops": 100.0 * m}
    if kind == "query_exact":
        return {"bytes": 28.0 * m, "flops": 80.0 * m}
    if kind == "exact_step":
        return {"bytes": 48.0 * n + 32.0 * m, "flops": 2 * solve + 2 * 27.0 * 8 * n + 80.0 * m}
    if kind == "shape":
        return {"bytes": 12.0 * n + 28.0 * m, "flops": forward["flops"] + solve + 27.0 * 8 * n + 200.0 * m}
    extra = 4.0 * cells if kind == "grid_step" else 20.0 * m
    return {"bytes": forward["bytes"] + 24.0 * n + extra,
            "flops": forward["flops"] + solve + 27.0 * 8 * n + 60.0 * m}


def tolerance(case):
    """About four times the error measured against `exact`.  phi and its sums
    are good to a few 1e-7; unit normals divide by |grad phi|, which vanishes
    on the medial axis, so single nodes there amplify the rounding ("max").
    The direction (q - y) / |q - y| of an exact query is the rounding of
    q - y over the distance, so queries next to the surface (a few per
    million within 1e-6 of it) carry the whole error: 2.5e-4 measured in the
    adjoint's sums.  Interpolated normals of the shape workload vanish between
    opposite ones and its points are 32-bit (6e-5 measured)."""
    kind = case["kind"]
    if kind == "normals":
        return {"rel": 1e-6, "max": 1e-3}
    if kind in ("query_exact", "exact_step"):
        return {"rel": 1e-3, "max": 0.99}
    if kind == "shape":
        return {"rel": 2.5e-4, "max": 0.1}
    return {"rel": 1e-5, "max": 0.02}


# ---------------------------------------------------------------- 64-bit restatement
def _spread(p, res):
    """Cells [n, 27, 3] around each point's own and their splat weights."""
    u = p * res
    own = torch.floor(u.detach()).long().clamp(0, res - 1)
    o = torch.tensor([(x, y, z) for z in (-1, 0, 1) for y in (-1, 0, 1) for x in (-1, 0, 1)], device=p.device)
    cells = own[:, None] + o
    f = 0.5 * (1 - (u[:, None] - (cells + 0.5)).abs() / 2).clamp(min=0)
    a = f.prod(2)
    a = torch.where((o == 0).all(1), torch.full_like(a, 0.5), a)
    a = torch.where(((cells >= 0) & (cells < res)).all(2), a, torch.zeros_like(a))
    return cells.clamp(0, res - 1), a / a.sum(1, keepdim=True)


def _flat(c, res):
    return (c[..., 2] * res + c[..., 1]) * res + c[..., 0]


def _mirrored(x, ax):
    """x at the lower and the upper neighbour along an axis, the walls mirrored."""
    n = x.shape[ax]
    i = torch.arange(n, device=x.device)
    return x.index_select(ax, (i - 1).clamp(min=0)), x.index_select(ax, (i + 1).clamp(max=n - 1))


def _mass(x, ax):
    lo, hi = _mirrored(x, ax)
    return 2 / 3 * x + (lo + hi) / 6


def _indicator(p, nrm, res, galerkin):
    """chi on the grid [z, y, x]: splat, divergence, Poisson solve."""
    cells, a = _spread(p, res)
    V = torch.zeros(res ** 3, 3, device=p.device, dtype=F64)
    V = V.index_add(0, _flat(cells, res).reshape(-1), (a[..., None] * nrm[:, None]).reshape(-1, 3))
    V = V.reshape(res, res, res, 3)
    b = 0
    for xi in range(3):
        ax = 2 - xi
        v = V[..., xi]
        face = 0.5 * (v.narrow(ax, 0, res - 1) + v.narrow(ax, 1, res - 1))
        pad = torch.zeros_like(v.narrow(ax, 0, 1))
        face = torch.cat([pad, face, pad], ax)
        t = face.narrow(ax, 1, res) - face.narrow(ax, 0, res)
        for other in range(3):
            if galerkin and other != ax:
                t = _mass(t, other)
        b = b + t
    k = torch.arange(res, device=p.device, dtype=F64)
    Q = torch.cos(math.pi * k[:, None] * (k[None] + 0.5) / res) * math.sqrt(2 / res)
    Q[0] *= math.sqrt(0.5)
    s = 4 * torch.sin(math.pi * k / (2 * res)) ** 2
    sx, sy, sz = s[None, None], s[None, :, None], s[:, None, None]
    if galerkin:
        mx, my, mz = 1 - sx / 6, 1 - sy / 6, 1 - sz / 6
        lam = -(sz * my * mx + mz * sy * mx + mz * my * sx)
    else:
        lam = -(sx + sy + sz)
    lam[0, 0, 0] = math.inf
    h = torch.einsum("kz,ly,mx,zyx->klm", Q, Q, Q, b) / lam
    return torch.einsum("kz,ly,mx,klm->zyx", Q, Q, Q, h)


def _corners(q, res):
    """The 8 grid nodes around q (clamped into the node hull) and their weights."""
    u = (q * res - 0.5).clamp(0, res - 1)
    i = torch.floor(u.detach()).long().clamp(max=res - 2)
    t = u - i
    bits = torch.tensor([(c & 1, c >> 1 & 1, c >> 2 & 1) for c in range(8)], device=q.device)
    w = torch.where(bits[None] == 1, t[:, None], 1 - t[:, None]).prod(2)
    return _flat(i[:, None] + bits, res), w


@functools.lru_cache(maxsize=1)
def _cases_of_a_cube():
    """Triangles (cube edge ids) of the 256 corner patterns, and each edge's
    (axis, lower corner, upper corner).  Edges 0-3 run along x, 4-7 along y,
    8-11 along z.  On every face the crossed edges are joined so that the
    inside corners (each alone on a face with two diagonal ones) lie to the
    right seen from outside; the loops are fanned from their lowest edge."""
    xyz = np.array([(k & 1, k >> 1 & 1, k >> 2 & 1) for k in range(8)])
    edges = []
    for axis in range(3):
        for side in range(4):
            lower = [k for k in range(8) if [xyz[k][i] for i in range(3) if i != axis] == [side & 1, side >> 1]
                     and xyz[k][axis] == 0]
            edges.append((axis, lower[0], lower[0] + (1 << axis)))
    out = []
    for pattern in range(256):
        inside = [pattern >> k & 1 for k in range(8)]
        cut = [e for e, (_, lo, hi) in enumerate(edges) if inside[lo] != inside[hi]]
        after = {}
        for axis in range(3):
            for side in (0, 1):
                outward = np.eye(3)[axis] * (2 * side - 1)
                here = [k for k in range(8) if xyz[k][axis] == side]
                on = [e for e in cut if edges[e][1] in here and edges[e][2] in here]
                wet = [k for k in here if inside[k]]
                groups = [wet] if len(on) == 2 else [[k] for k in wet] if len(on) == 4 else []
                for group in groups:
                    a, b = on if len(on) == 2 else [e for e in on if group[0] in edges[e][1:]]
                    pa, pb = ((xyz[edges[e][1]] + xyz[edges[e][2]]) / 2 for e in (a, b))
                    if np.dot(np.cross(outward, pb - pa), xyz[group].mean(0) - (pa + pb) / 2) > 0:
                        a, b = b, a
                    after[a] = b
        tris, seen = [], set()
        for e in cut:
            loop = []
            while e not in seen:
                seen.add(e)
                loop.append(e)
                e = after[e]
            tris += [(loop[0], loop[k], loop[k + 1]) for k in range(1, len(loop) - 1)]
        out.append(tris)
    return out, edges


def _mesh(chi, c):
    """Triangles [T, 3, 3] of chi = c, differentiable in chi and c."""
    res = chi.shape[0]
    inside = chi.detach() < c.detach()
    m, code = res - 1, 0
    for k in range(8):
        x, y, z = k & 1, k >> 1 & 1, k >> 2 & 1
        code = code + (inside[z:z + m, y:y + m, x:x + m].long() << k)
    table, edges = _cases_of_a_cube()
    nodes, axes = [], []
    for pattern in range(1, 255):
        at = (code == pattern).nonzero() if table[pattern] else None
        if at is None or not len(at):
            continue
        base = at.flip(1)
        tri = table[pattern]
        low = torch.tensor([[[edges[e][1] >> b & 1 for b in range(3)] for e in t] for t in tri], device=chi.device)
        nodes.append((base[:, None, None] + low[None]).reshape(-1, 3, 3))
        axes.append(torch.tensor([[edges[e][0] for e in t] for t in tri], device=chi.device).repeat(len(base), 1, 1)
                    .reshape(-1, 3))
    node, step = torch.cat(nodes), torch.nn.functional.one_hot(torch.cat(axes), 3)
    c1, c2 = (chi.reshape(-1)[_flat(v, res)] for v in (node, node + step))
    return (node + 0.5 + ((c - c1) / (c2 - c1))[..., None] * step) / res


def _closest(q, tri, cell):
    """Index of each point's closest triangle and the weights of its closest
    point's second and third vertex; points are taken in cells of the given
    edge, against the triangles that some point of the cell may be closest to."""
    a, ab, ac = tri[:, 0], tri[:, 1] - tri[:, 0], tri[:, 2] - tri[:, 0]
    mid = tri.mean(1)
    rad = (tri - mid[:, None]).norm(dim=2).max(1).values
    per = torch.stack([(ab * ab).sum(1), (ab * ac).sum(1), (ac * ac).sum(1)])
    key = torch.floor((q + 1) / cell).long()
    key = (key[:, 2] * 4096 + key[:, 1]) * 4096 + key[:, 0]
    key, order = key.sort()
    counts = torch.unique_consecutive(key, return_counts=True)[1].tolist()
    idx = torch.empty(len(q), device=q.device, dtype=torch.long)
    vw = torch.empty(len(q), 2, device=q.device, dtype=F64)
    begin = 0
    for count in counts:
        at = order[begin:begin + count]
        begin += count
        p = q[at]
        lo, hi = p.min(0).values, p.max(0).values
        p0, e = (lo + hi) / 2, (hi - lo) / 2
        d0 = ((mid - p0) ** 2).sum(1)
        best = d0.argmin()
        # |p - mid| <= |p - y| + rad for some p of the box (y: the middle closest to its centre)
        room = 2 * ((mid - mid[best]).abs() * e).sum(1) + 2 * rad * (d0[best].sqrt() + e.norm()) + rad * rad
        near = (d0 - d0[best] <= room * (1 + 1e-9) + 1e-15).nonzero()[:, 0]
        for part in p.split(max(1, 40_000_000 // max(1, len(near)))):
            A, B, C = a[near], ab[near], ac[near]
            e00, e01, e11 = per[:, near]
            s = (part * part).sum(1)[:, None] - 2 * part @ A.T + (A * A).sum(1)
            d1, d2 = part @ B.T - (A * B).sum(1), part @ C.T - (A * C).sum(1)

            def at_weights(v, w):
                return s - 2 * v * d1 - 2 * w * d2 + v * v * e00 + 2 * v * w * e01 + w * w * e11

            zero = torch.zeros_like(s)
            tb = ((d2 - d1 - e01 + e00) / (e00 - 2 * e01 + e11)).clamp(0, 1)
            det = e00 * e11 - e01 * e01
            v, w = (e11 * d1 - e01 * d2) / det, (e00 * d2 - e01 * d1) / det
            ok = (v >= 0) & (w >= 0) & (v + w <= 1)
            tried = [((d1 / e00).clamp(0, 1), zero), (zero, (d2 / e11).clamp(0, 1)), (1 - tb, tb),
                     (torch.where(ok, v, zero), torch.where(ok, w, zero))]
            least = functools.reduce(torch.minimum, [torch.nan_to_num(at_weights(*x), nan=math.inf) for x in tried])
            j = least.argmin(1)
            row = torch.arange(len(part), device=q.device)
            d = torch.stack([torch.nan_to_num(at_weights(*x)[row, j], nan=math.inf) for x in tried])
            which = d.argmin(0)
            pick = torch.stack([torch.stack([x[0][row, j], x[1][row, j]], 1) for x in tried])[which, row]
            rows = at[:len(part)]
            at = at[len(part):]
            idx[rows], vw[rows] = near[j], pick
    return idx, vw


def _distance(q, tri, cell):
    """Distance to the mesh, differentiable in q and the vertices."""
    with torch.no_grad():
        idx, vw = _closest(q.detach(), tri.detach(), cell)
    t = tri[idx]
    y = t[:, 0] + vw[:, :1] * (t[:, 1] - t[:, 0]) + vw[:, 1:] * (t[:, 2] - t[:, 0])
    return (q - y).norm(dim=1)


def _inside(q, tri):
    """Whether the closed mesh winds around q (sum of solid angles)."""
    out = []
    for p in q.split(max(1, 20_000_000 // max(1, len(tri)))):
        A, B, C = (tri[None, :, k] - p[:, None] for k in range(3))
        a, b, c = A.norm(dim=2), B.norm(dim=2), C.norm(dim=2)
        det = (A * torch.linalg.cross(B, C)).sum(2)
        den = a * b * c + (A * B).sum(2) * c + (B * C).sum(2) * a + (C * A).sum(2) * b
        out.append(2 * torch.atan2(det, den).sum(1).abs() > 2 * math.pi)
    return torch.cat(out)


def _unit_normals(phi):
    res = phi.shape[0]
    grads = []
    for ax in (2, 1, 0):
        def at(i, k):
            return phi.narrow(ax, i, k)
        inner = (at(2, res - 2) - at(0, res - 2)) / 2
        first = (-3 * at(0, 1) + 4 * at(1, 1) - at(2, 1)) / 2
        last = (3 * at(res - 1, 1) - 4 * at(res - 2, 1) + at(res - 3, 1)) / 2
        grads.append(torch.cat([first, inner, last], ax))
    g = torch.stack(grads)
    return g / g.norm(dim=0, keepdim=True)


def _surface(p, nrm, res, galerkin):
    chi = _indicator(p, nrm, res, galerkin)
    node, w = _corners(p, res)
    c = (chi.reshape(-1)[node] * w).sum(1).mean()
    return chi, c, _mesh(chi, c)


def _phi_grid(chi, c, tri):
    res = chi.shape[0]
    z, y, x = torch.meshgrid(*[torch.arange(res, device=chi.device)] * 3, indexing="ij")
    nodes = (torch.stack([x, y, z], -1).reshape(-1, 3).to(F64) + 0.5) / res
    sign = torch.where(chi.detach() < c.detach(), -1.0, 1.0)
    return sign * _distance(nodes, tri, 8 / res).reshape(res, res, res)


def _harmonics(lmax, u):
    """Orthonormal real spherical harmonics (no Condon-Shortley phase) at unit
    u, index l*l + l + m, as polynomials in the Cartesian components."""
    x, y, z = u.unbind(1)
    cs = [(torch.ones_like(x), torch.zeros_like(x))]
    for _ in range(lmax):
        c, s = cs[-1]
        cs.append((x * c - y * s, x * s + y * c))
    out = [None] * (lmax + 1) ** 2
    for m in range(lmax + 1):
        q = {m: torch.full_like(z, float(math.prod(range(1, 2 * m, 2))))}
        for l in range(m, lmax + 1):
            if l > m:
                q[l] = ((2 * l - 1) * z * q[l - 1] - (l + m - 1) * q.get(l - 2, torch.zeros_like(z))) / (l - m)
            k = math.sqrt((2 * l + 1) / (4 * math.pi) * math.factorial(l - m) / math.factorial(l + m))
            k *= math.sqrt(2) if m else 1
            out[l * l + l + m] = k * q[l] * cs[m][0]
            if m:
                out[l * l + l - m] = k * q[l] * cs[m][1]
    return torch.stack(out, 1)


def _harmonic_body(theta, dirs, lmax):
    """Points and normals of r(u) = 0.3 + sum theta_k Y_k(u)."""
    u = dirs.detach().requires_grad_()
    r = 0.3 + _harmonics(lmax, u) @ theta
    (g,) = torch.autograd.grad(r.sum(), u, create_graph=True)
    g = g - (g * dirs).sum(1, keepdim=True) * dirs
    nrm = dirs - g / r[:, None]
    return CENTRE + r[:, None] * dirs, nrm / nrm.norm(dim=1, keepdim=True)


def _plane_normals(points, outward, radius, eps):
    """Distance-weighted PCA normals, signed like `outward`; members are taken
    by the 32-bit test the library documents."""
    p32, p = points, points.to(F64)
    key = torch.floor(p / (radius / 2)).long()
    key, order = ((key[:, 2] * 4096 + key[:, 1]) * 4096 + key[:, 0]).sort()
    counts = torch.unique_consecutive(key, return_counts=True)[1].tolist()
    out = torch.empty_like(p)
    begin = 0
    r2 = torch.tensor(radius, device=p.device, dtype=torch.float32) ** 2
    for count in counts:
        cell = order[begin:begin + count]
        begin += count
        lo, hi = p[cell].min(0).values - 1.001 * radius, p[cell].max(0).values + 1.001 * radius
        near = ((p >= lo) & (p <= hi)).all(1).nonzero()[:, 0]
        for at in cell.split(max(1, 20_000_000 // len(near))):
            d = p32[near][None] - p32[at][:, None]
            member = (d[..., 0] * d[..., 0] + d[..., 1] * d[..., 1]) + d[..., 2] * d[..., 2] <= r2
            del d
            w = torch.where(member, 1 / (torch.cdist(p[at], p[near], compute_mode="donot_use_mm_for_euclid_dist")
                                         + eps), 0.0)
            W = w.sum(1)
            x = p[near] - p[at].mean(0)
            bar = w @ x / W[:, None]
            second = (w @ (x[:, :, None] * x[:, None]).reshape(-1, 9)).reshape(-1, 3, 3) / W[:, None, None]
            out[at] = torch.linalg.eigh(second - bar[:, :, None] * bar[:, None])[1][:, :, 0]
    return out * torch.sign((out * outward).sum(1, keepdim=True))


def exact(case, seed):
    kind, res = case["kind"], case.get("res", 0)
    x = _inputs(case, seed)
    if kind == "normals":
        return _plane_normals(x["points"], x["normals"].to(F64), case["radius"], 1e-3 * case["radius"])
    if res > 130 or kind == "moving":
        return None  # the nearest triangle of every node takes too long here
    x = {k: v.to(F64) for k, v in x.items()}
    if kind == "shape":
        theta = x["theta"].requires_grad_()
        p, nrm = _harmonic_body(theta, x["dirs"], case["lmax"])
    else:
        p, nrm = x["points"].requires_grad_(), x["normals"].requires_grad_()
    chi, c, tri = _surface(p, nrm, res, case["galerkin"])
    if kind in ("query_exact", "exact_step"):
        q = x["q"].requires_grad_()
        node, _ = _corners(q.detach(), res)
        wet = (chi < c).reshape(-1)[node]
        inside = wet[:, 0].clone()
        mixed = wet.any(1) & ~wet.all(1)
        if mixed.any():
            inside[mixed] = _inside(q.detach()[mixed], tri.detach())
        phi = torch.where(inside, -1.0, 1.0) * _distance(q, tri, 8 / res)
        if kind == "query_exact":
            return phi.detach(), torch.autograd.grad(phi.sum(), q)[0]
        return (phi.detach(), *torch.autograd.grad(phi, (p, nrm, q), x["seed_q"]))
    phi = _phi_grid(chi, c, tri)
    unit = _unit_normals(phi)
    if kind == "forward":
        return phi.detach(), unit.detach()
    if kind == "grid_step":
        return (phi.detach(), unit.detach(), *torch.autograd.grad(phi, (p, nrm), x["seed_grid"]))
    node, w = _corners(x["q"], res)
    phi_q = (phi.reshape(-1)[node] * w).sum(1)
    if kind == "step":
        return (phi.detach(), unit.detach(), phi_q.detach(), *torch.autograd.grad(phi_q, (p, nrm), x["seed_q"]))
    unit_q = (unit.detach().reshape(3, -1)[:, node] * w.detach()).sum(2).T
    unit_q = unit_q / unit_q.norm(dim=1, keepdim=True)
    if kind == "query":
        return phi_q.detach(), unit_q
    loss = ((phi_q - ((x["q"] - CENTRE).norm(dim=1) - 0.3)) ** 2).mean()
    (dtheta,) = torch.autograd.grad(loss, theta)
    return phi_q.detach(), unit_q, dtheta
