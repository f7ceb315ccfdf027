"""The calls whose speed this repository is measured by: manifold tracing,
certification, batched and served tracing, batch triangulation and plain
evaluation of the decision function, each through the Python entry points of
``paper_2406_04795_gb300.api`` on seeded synthetic problems.

``listed()`` gives the cases, ``draw(rng)`` further ones of the same ranges,
``prepare(case, seed)`` what a program holds before the call, ``run(state)`` the
call, ``work(case)`` the bytes and operations it cannot do without and
``exact(case, seed)`` its floating-point results in 64 bits by plain torch.

Problems: support vectors uniform in [-pi, pi]^d at the density of the
repository's own workloads (64 vectors in d = 3, 2048 in d = 5, 8192 in d = 6),
a serial DH arm with capsule links among boxes and spheres, twice the capacities
of ``pipeline.sizing_for``.  A case fixes its manifold; a seed gives the inputs of
one instance of it: the axes permuted, C-space inverted or not (the
triangulation and the box are symmetric under both), the support vectors in
another order, f scaled, and another robot among other obstacles, so that every
input array differs while the traced set keeps its size.  Proofs ask for the
sorted output; the batched, served and subdivided calls have no such option, so
their results are put in key order after the call, as a program that compares
or stores them has to.
"""
import itertools
import math

import numpy as np
import torch

from paper_2406_04795_gb300 import mf
from paper_2406_04795_gb300 import pipeline
from paper_2406_04795_gb300 import workloads as W
from paper_2406_04795_gb300.api import Context

PRECISION = {"fp64": mf.MF_FP64, "bf16": mf.MF_MIXED_BF16, "fp32": mf.MF_MIXED_FP32}
GAMMA = {3: 2.0, 4: 4.0, 5: 4.0, 6: 6.0}
# traced edges at the reference lambda, cells per edge and traced edges per
# cell of the random problems (measured; the traced set grows as
# lambda^-(d-1)), for the work estimates
EDGES_REF = {3: (4.0e4, 0.1), 4: (4.4e5, 0.08), 5: (1.0e8, 0.05), 6: (2.0e6, 0.2)}
CELLS_PER_EDGE = {3: 1.55, 4: 3.2, 5: 8.3, 6: 29.0}
EDGES_PER_CELL = {3: 3.3, 4: 4.9, 5: 6.6, 6: 7.8}
SHELL_EDGES = {4: 1.0e5, 5: 3.5e5}  # per shell of a batched trace


def listed():
    return [
        # a planner asks for f at a handful of configurations: a launch-bound call
        dict(name="eval_small", kind="eval", d=3, n_sv=64, n=1000, precision="fp64"),
        # f over a sampled C-space for a 5-DoF arm's manifold, full precision
        dict(name="eval_fp64", kind="eval", d=5, n_sv=2048, n=200003, precision="fp64"),
        # the same for a 6-DoF arm and its larger model, mixed precision
        dict(name="eval_mixed", kind="eval", d=6, n_sv=8192, n=100000, precision="fp32"),
        # collision check of a sampled C-space: sphere robot with link capsules
        # among boxes, spheres and cylinders, no cells
        dict(name="certify_points", kind="certify", d=6, n=500009, n_obs=18, spheres=3),
        # the smallest proof: 3-DoF planar arm, thousands of edges, many short levels
        dict(name="proof_d3", kind="proof", d=3, n_sv=64, lam=0.1, n_seeds=1, precision="fp64"),
        # an ordinary 4-DoF proof on the FP32 mixed path, a ragged model size
        dict(name="proof_d4_fp32", kind="proof", d=4, n_sv=333, lam=0.07, n_seeds=8,
             precision="fp32"),
        # the ordinary 5-DoF proof, coarse lattice
        dict(name="proof_d5", kind="proof", d=5, n_sv=2048, lam=0.15, n_seeds=16,
             precision="fp64"),
        # the 5-DoF proof at a fine lattice: the largest call
        dict(name="proof_d5_fine", kind="proof", d=5, n_sv=2048, lam=0.08, n_seeds=16,
             precision="fp64"),
        # the 6-DoF proof on the tensor-core path
        dict(name="proof_d6_bf16", kind="proof", d=6, n_sv=8192, lam=0.22, n_seeds=64,
             precision="bf16"),
        # independent manifolds traced in one call
        dict(name="batch", kind="batch", d_lo=4, d_hi=5, n_traces=8, sv_lo=256, sv_hi=8192,
             precision="bf16"),
        # requests through the proof server, from submission to the fetched results
        dict(name="served", kind="served", d_lo=4, d_hi=4, n_traces=4, sv_lo=512, sv_hi=4096,
             precision="fp64"),
        # batch triangulation: coarse trace, every crossing n-simplex subdivided
        dict(name="subdiv_d4", kind="subdiv", d=4, n_sv=333, lam=0.06, k=2, n_seeds=8,
             precision="fp64"),
    ]


def _log(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def _model(rng, d):
    """A model size: a third of the repository's density up to all of it."""
    top = {3: 64, 4: 400, 5: 2048, 6: 8192}[d]
    return int(_log(rng, top / 3, top))


def draw(rng):
    kind = rng.choice(["eval", "certify", "proof", "proof", "proof", "proof", "batch", "served",
                       "subdiv"])
    if kind == "eval":
        d = rng.randint(3, 6)
        return dict(kind=kind, d=d, n_sv=int(_log(rng, 64, 8192)), n=int(_log(rng, 1000, 200000)),
                    precision=rng.choice(["fp64", "fp32"]))
    if kind == "certify":
        return dict(kind=kind, d=rng.randint(3, 6), n=int(_log(rng, 1000, 500000)),
                    n_obs=rng.randint(4, 18), spheres=rng.randint(0, 3))
    if kind == "proof":
        d = rng.randint(3, 6)
        lo, hi = {3: (0.06, 0.2), 4: (0.06, 0.2), 5: (0.09, 0.3), 6: (0.23, 0.5)}[d]
        return dict(kind=kind, d=d, n_sv=_model(rng, d), lam=round(_log(rng, lo, hi), 4),
                    n_seeds=1 if d == 3 else rng.randint(1, 64),
                    precision=rng.choice(["fp64", "bf16", "fp32"]))
    if kind == "subdiv":
        d = rng.randint(3, 4)
        return dict(kind=kind, d=d, n_sv=_model(rng, d), lam=round(_log(rng, 0.07, 0.15), 4),
                    k=rng.randint(2, 3), n_seeds=1 if d == 3 else rng.randint(1, 16),
                    precision=rng.choice(["fp64", "fp32"]))
    d_hi = rng.randint(4, 5)
    return dict(kind=kind, d_lo=4, d_hi=d_hi, n_traces=rng.randint(2, 6),
                sv_lo=256 if kind == "batch" else 512, sv_hi=int(_log(rng, 1024, 8192)),
                precision=rng.choice(["fp64", "bf16", "fp32"]))


# ---------------------------------------------------------------------------
# Inputs
# ---------------------------------------------------------------------------
_held = {}


def _context():
    """The one context a program keeps: its resident tables serve every call."""
    if "ctx" not in _held:
        _held["ctx"] = Context(0, 120 << 30)
    return _held["ctx"]


def _server():
    """A long-lived proof server on a context of its own."""
    if "server" not in _held:
        _held["server_ctx"] = Context(0, 40 << 30)
        _held["server"] = _held["server_ctx"].server(max_slots=16, hbm_bytes=32 << 30)
    return _held["server"]


def _dev(x, dtype=torch.float64):
    return torch.as_tensor(np.ascontiguousarray(x)).to(device="cuda", dtype=dtype)


def _f(x, sv, alpha, gamma, b):
    """The decision function at x [n, d] in 64 bits (support vectors in chunks)."""
    out = torch.full((x.shape[0],), float(b), dtype=torch.float64, device=x.device)
    step = max(1, int(4e7) // max(1, sv.shape[0]))
    for a in range(0, x.shape[0], step):
        r2 = torch.zeros((min(step, x.shape[0] - a), sv.shape[0]), dtype=torch.float64,
                         device=x.device)
        for k in range(sv.shape[1]):
            r2 += (x[a:a + step, k, None] - sv[None, :, k]).square_()
        out[a:a + step] += r2.mul_(-gamma).exp_() @ alpha
    return out


def _seeds(gen, sv, alpha, gamma, b, n_seeds):
    """Points with f = 0: from free-space vectors with f < 0 outwards until
    f >= 0, then bisection (the manifold sampler's stand-in)."""
    d = sv.shape[1]
    free = sv[alpha < 0]
    free = free[_f(free, sv, alpha, gamma, b) < 0]
    n = 8 * n_seeds
    a = free[torch.randint(free.shape[0], (n,), generator=gen, device="cuda")]
    u = torch.randn((n, d), generator=gen, dtype=torch.float64, device="cuda")
    u /= u.norm(dim=1, keepdim=True)
    t = torch.arange(1, 101, dtype=torch.float64, device="cuda") * 0.05
    p = a[:, None, :] + t[None, :, None] * u[:, None, :]
    inside = (p.abs() <= math.pi).all(2)
    up = (_f(p.reshape(-1, d), sv, alpha, gamma, b).reshape(n, -1) >= 0) & inside
    first = torch.where(up.any(1), up.float().argmax(1), torch.full((n,), -1, device="cuda"))
    stays = inside.long().cumprod(1).bool()
    ok = (first >= 0) & stays.gather(1, first.clamp(min=0)[:, None])[:, 0]
    a, u, first = a[ok][:n_seeds], u[ok][:n_seeds], first[ok][:n_seeds]
    lo, hi = t[first] - 0.05, t[first]
    for _ in range(60):
        m = 0.5 * (lo + hi)
        pos = _f(a + m[:, None] * u, sv, alpha, gamma, b) >= 0
        hi, lo = torch.where(pos, m, hi), torch.where(pos, lo, m)
    return a + (0.5 * (lo + hi))[:, None] * u


def _aabb(centers):
    pose = np.zeros((centers.shape[0], 12))
    pose[:, [0, 4, 8]] = 1.0
    pose[:, 9:] = centers
    return pose


def _base(*values):
    """The seed of the manifold that a case stands for."""
    return int(sum((i + 1) * 7919 * round(1e4 * v) for i, v in enumerate(values))) % (1 << 31)


def _instance(w, seed):
    """The seed's instance of a trace: axes permuted, C-space inverted or not,
    support vectors reordered, f scaled."""
    rng = np.random.default_rng(seed)
    axes, sign, scale = rng.permutation(w.d), rng.choice([-1.0, 1.0]), rng.uniform(0.8, 1.25)
    order = torch.from_numpy(rng.permutation(w.sv.shape[0])).cuda()
    ax = torch.from_numpy(axes).cuda()
    w.sv, w.alpha, w.b = sign * w.sv[order][:, ax], scale * w.alpha[order], scale * w.b
    w.seeds, w.offset = sign * w.seeds[:, ax], sign * w.offset[axes]
    return w


def _problem(case, seed):
    """One tracing problem: a workload whose arrays are on the GPU."""
    d, n_sv, lam = case["d"], case["n_sv"], case.get("lam", 0.1)
    gen = torch.Generator(device="cuda").manual_seed(_base(d, n_sv, lam, case.get("n_seeds", 1)))
    rng = np.random.default_rng(seed)
    sv = (torch.rand((n_sv, d), generator=gen, dtype=torch.float64, device="cuda") * 2 - 1) * math.pi
    alpha = torch.randn(n_sv, generator=gen, dtype=torch.float64, device="cuda")
    gamma = GAMMA[d]
    if d == 3:  # a zero of f at the origin by construction
        b = -float(alpha @ torch.exp(-gamma * sv.square().sum(1)))
        seeds = torch.zeros((1, d), dtype=torch.float64, device="cuda")
        dh = np.zeros((d, 4))
        dh[:, 2] = 1.0
        radius = np.full(d, 0.05)
        centers = np.zeros((4, 3))
        centers[:, :2] = rng.uniform(-2.5, 2.5, size=(4, 2))
        types, dims = np.zeros(4, np.int32), 2.0 * rng.uniform(0.1, 0.5, size=(4, 3))
    else:
        free = torch.rand(n_sv, generator=gen, device="cuda") < 0.3
        alpha = torch.where(free, -alpha.abs(), alpha.abs())
        b = 0.6
        seeds = _seeds(gen, sv, alpha, gamma, b, case.get("n_seeds", 1))
        dh, radius = W._dh_arm(rng, d, 0.04)
        reach = float(dh[:, 2].sum())
        n_box, n_sph = (10, 10) if d == 6 else (12, 0)
        centers = W._ball(rng, n_box + n_sph, reach)
        types = np.array([W.BOX] * n_box + [W.SPHERE] * n_sph, np.int32)
        dims = 2.0 * rng.uniform(0.05, 0.3, size=(n_box + n_sph, 3))
        dims[n_box:] = 0.0
        dims[n_box:, 0] = rng.uniform(0.05, 0.25, size=n_sph)
    lo, hi = np.full(d, -math.pi), np.full(d, math.pi)
    w = W.Workload("d%d_%dsv" % (d, n_sv), d, sv, alpha, gamma, b, lam, W.lattice_offset(d, lam),
                   lo, hi, seeds, _dev(dh), _dev(radius), _dev(types, torch.int32),
                   _dev(_aabb(centers)), _dev(dims))
    return _instance(w, seed)


def _shells(case, seed):
    """The traces of a batched or served call, d and sizes mixed."""
    rng = np.random.default_rng(_base(case["d_lo"], case["d_hi"], case["n_traces"], case["sv_hi"]))
    out = []
    for t in range(case["n_traces"]):
        d = case["d_lo"] + t % (case["d_hi"] - case["d_lo"] + 1)
        n_sv = int(round(math.exp(rng.uniform(math.log(case["sv_lo"]), math.log(case["sv_hi"])))))
        w = W.shell_trace(rng, d, n_sv, float(rng.uniform(0.03, 0.1)), int(rng.integers(1, 9)),
                          n_free=int(rng.integers(1, 3)))
        w.sv, w.alpha, w.seeds = _dev(w.sv), _dev(w.alpha), _dev(w.seeds)
        out.append(_instance(w, seed + 1000 * t))
    return out


def _sampled_scene(case, seed):
    """A random arm with link spheres among boxes, spheres and cylinders, and
    uniformly sampled configurations."""
    rng = np.random.default_rng(seed)
    gen = torch.Generator(device="cuda").manual_seed(seed)
    d, n_obs = case["d"], case["n_obs"]
    dh, radius = W._dh_arm(rng, d, 0.04)
    dh[:, 0] = rng.uniform(-1, 1, d)
    reach = float(dh[:, 2].sum())
    types = np.arange(n_obs, dtype=np.int32) % 3
    pose = _aabb(rng.uniform(-reach, reach, size=(n_obs, 3)))
    for i in np.flatnonzero(types != W.SPHERE):
        q, _ = np.linalg.qr(rng.normal(size=(3, 3)))
        pose[i, :9] = (q if np.linalg.det(q) > 0 else q[:, ::-1]).reshape(-1)
    dims = np.zeros((n_obs, 3))
    box, sph, cyl = types == 0, types == 1, types == 2
    dims[box] = rng.uniform(0.1, 0.5, size=(box.sum(), 3))
    dims[sph, 0] = rng.uniform(0.05, 0.25, sph.sum())
    dims[cyl, 0] = rng.uniform(0.03, 0.2, cyl.sum())
    dims[cyl, 1] = rng.uniform(0.2, 0.9, cyl.sum())
    spheres = None
    if case["spheres"]:
        link = np.repeat(np.arange(d), case["spheres"]).astype(np.int32)
        centre = np.stack([-rng.uniform(0, 1, link.size) * dh[link, 2],
                           rng.uniform(-0.03, 0.03, link.size),
                           rng.uniform(-0.03, 0.03, link.size)], 1)
        spheres = (_dev(link, torch.int32), _dev(centre), _dev(rng.uniform(0.03, 0.08, link.size)))
    q = torch.rand((case["n"], d), generator=gen, dtype=torch.float64, device="cuda")
    return dict(dh=_dev(dh), radius=_dev(radius), types=_dev(types, torch.int32), pose=_dev(pose),
                dims=_dev(dims), spheres=spheres, points=(q * 2 - 1) * math.pi)


def _points(case, w, seed):
    """Query configurations: half uniform, half close to support vectors."""
    gen = torch.Generator(device="cuda").manual_seed(seed + 1)
    n, d = case["n"], case["d"]
    q = (torch.rand((n, d), generator=gen, dtype=torch.float64, device="cuda") * 2 - 1) * math.pi
    near = w.sv[torch.randint(w.sv.shape[0], (n,), generator=gen, device="cuda")]
    near = near + 0.2 * torch.randn((n, d), generator=gen, dtype=torch.float64, device="cuda")
    return torch.where((torch.arange(n, device="cuda") % 2 == 0)[:, None], q, near)


def prepare(case, seed):
    state = dict(case=case, precision=PRECISION[case.get("precision", "fp64")])
    kind = case["kind"]
    if kind == "certify":
        state.update(ctx=_context(), scene=_sampled_scene(case, seed))
    elif kind in ("batch", "served"):
        state["traces"] = _shells(case, seed)
        state["caps"] = [W.shell_capacity(w) for w in state["traces"]]
        if kind == "batch":
            state["ctx"] = _context()
        else:
            state["server"] = _server()
    else:
        w = _problem(case, seed)
        state.update(ctx=_context(), w=w)
        if kind == "eval":
            state["points"] = _points(case, w, seed)
        else:
            state["sizing"] = {k: 2 * v for k, v in pipeline.sizing_for(w).items()}
    return state


# ---------------------------------------------------------------------------
# The calls
# ---------------------------------------------------------------------------
def _lattice_key(y, rest):
    """Sorting key of lattice objects: sum(y), y_{d-2} .. y_0, then the columns
    of `rest` (the order of mf_trace's sorted output)."""
    y = y.long()
    d = y.shape[1]
    cols = [y.sum(1)] + [y[:, k] for k in range(d - 2, -1, -1)] + [r.long() for r in rest]
    key = torch.zeros_like(cols[0])
    for c in cols:
        lo = c.amin()
        key = key * (c.amax() - lo + 1) + (c - lo)
    return key


EDGE_FIELDS = ("edge_y", "edge_mask", "edge_f", "edge_t", "points")


def _in_order(r, cells):
    """A trace's result in key order."""
    if r["n_edges"] == 0:
        return {k: r[k] for k in EDGE_FIELDS + (("cell_y", "cell_perm", "cell_off", "cell_idx")
                                                if cells else ())}
    order = torch.argsort(_lattice_key(r["edge_y"], [r["edge_mask"]]))
    out = {k: r[k][order] for k in EDGE_FIELDS}
    if cells:
        perm = r["cell_perm"]
        corder = torch.argsort(_lattice_key(r["cell_y"], [perm[:, k] for k in range(perm.shape[1])]))
        rank = torch.empty_like(order)
        rank[order] = torch.arange(order.shape[0], device=order.device)
        first, n = r["cell_off"][:-1][corder], (r["cell_off"][1:] - r["cell_off"][:-1])[corder]
        off = torch.zeros_like(r["cell_off"])
        torch.cumsum(n, 0, out=off[1:])
        src = torch.repeat_interleave(first - off[:-1], n, output_size=r["n_cell_edges"])
        src += torch.arange(src.shape[0], device=src.device)
        out.update(cell_y=r["cell_y"][corder], cell_perm=perm[corder], cell_off=off,
                   cell_idx=rank[r["cell_idx"][src]])
    return out


COUNTS = ("n_vertices", "n_boundary", "n_near_zero", "n_dead_seeds", "levels")


def _joined(results, cells=True):
    """The results of several traces, each field as one array."""
    parts = [_in_order(r, cells) for r in results]
    out = {k: torch.cat([p[k].reshape(-1) for p in parts]) for k in parts[0]}
    out["counts"] = np.array([[r[k] for k in COUNTS] for r in results], np.int64)
    return out


def _proof(s):
    w, ctx = s["w"], s["ctx"]
    r = ctx.trace(w.sv, w.alpha, w.gamma, w.b, w.lam, w.offset, w.lo, w.hi, w.seeds,
                  precision=s["precision"], sort=True, **s["sizing"])
    c = ctx.certify_ex(w.dh, w.radius, w.obs_type, w.obs_pose, w.obs_dims, r["points"],
                       r["cell_off"], r["cell_idx"], whole=True, slack=False)
    out = {k: r[k] for k in EDGE_FIELDS + ("cell_y", "cell_perm", "cell_off", "cell_idx")}
    out["counts"] = np.array([r[k] for k in COUNTS], np.int64)
    out.update({k: c[k] for k in ("verdict", "margin", "element", "cell_verdict", "cell_whole")
                if k in c})
    return out


def _certify(s):
    q = s["scene"]
    c = s["ctx"].certify_ex(q["dh"], q["radius"], q["types"], q["pose"], q["dims"], q["points"],
                            spheres=q["spheres"])
    return {k: c[k] for k in ("verdict", "margin", "element")}


def _serve(s):
    server = s["server"]
    ids = [server.submit(w, precision=s["precision"], **cap)
           for w, cap in zip(s["traces"], s["caps"])]
    got, left = {}, set(ids)
    while left:
        server.step()
        for rid in server.done():
            left.discard(rid)
            got[rid] = server.fetch(rid)
    return _joined([got[rid] for rid in ids])


def run(state):
    kind = state["case"]["kind"]
    if kind == "eval":
        w = state["w"]
        return state["ctx"].eval(w.sv, w.alpha, w.gamma, w.b, state["points"],
                                 precision=state["precision"])
    if kind == "certify":
        return _certify(state)
    if kind == "proof":
        return _proof(state)
    if kind == "batch":
        return _joined(state["ctx"].trace_batch(state["traces"],
                                                [state["precision"]] * len(state["traces"]),
                                                capacities=state["caps"]))
    if kind == "served":
        return _serve(state)
    r = state["ctx"].subdiv(state["w"], state["case"]["k"], precision=state["precision"],
                            **state["sizing"])
    out = _in_order(r, False)
    out["counts"] = np.array([r["n_vertices"], r["n_near_zero"], r["n_coarse_cells"], r["levels"],
                              r["n_dead_seeds"]], np.int64)
    return out


# ---------------------------------------------------------------------------
# What a call cannot do without
# ---------------------------------------------------------------------------
def _kept(d, n_sv, gamma, cut=20.0):
    """Expected support vectors near a point that its sum needs: those with
    gamma r^2 <= cut (about 1e-9 of a weight), in [-pi, pi]^d."""
    r = math.sqrt(cut / gamma)
    ball = math.pi ** (d / 2) / math.gamma(d / 2 + 1) * r ** d
    return max(1.0, min(1.0, ball / (2 * math.pi) ** d) * n_sv)


def _trace_work(d, n_sv, gamma, E, cells=True):
    per_edge = 4 * d + 4 + 16 + 8 + 8 * d
    per_cell = 5 * d + 8 + 8 * EDGES_PER_CELL[d]
    C = CELLS_PER_EDGE[d] * E if cells else 0
    # f at ~0.2 vertices and at one root per edge
    flops = 1.2 * E * _kept(d, n_sv, gamma) * (3 * d + 20)
    return n_sv * (d + 1) * 8 + E * per_edge + C * per_cell, flops


def work(case):
    kind = case["kind"]
    if kind == "eval":
        d, n, m = case["d"], case["n"], case["n_sv"]
        return dict(bytes=m * (d + 1) * 8 + n * (d + 1) * 8, flops=n * _kept(d, m, GAMMA[d]) * (3 * d + 20))
    if kind == "certify":
        d, n, el = case["d"], case["n"], case["d"] * (1 + case["spheres"])
        # the chain (30 operations a joint) and one distance bound per pair
        return dict(bytes=n * (8 * d + 11), flops=n * (40 * d + 40 * el * case["n_obs"]))
    if kind in ("batch", "served"):
        by = fl = 0.0
        for t in range(case["n_traces"]):
            d = case["d_lo"] + t % (case["d_hi"] - case["d_lo"] + 1)
            b, f = _trace_work(d, math.sqrt(case["sv_lo"] * case["sv_hi"]), 25.0, 1.5 * SHELL_EDGES[d])
            by, fl = by + b, fl + f
        return dict(bytes=by, flops=fl)
    d, m = case["d"], case["n_sv"]
    E0, lam0 = EDGES_REF[d]
    E = E0 * (lam0 / case["lam"]) ** (d - 1)
    b, f = _trace_work(d, m, GAMMA[d], E, cells=kind == "proof")
    if kind == "proof":  # and the certificate of every point and cell
        b += E * (8 * d + 11) + CELLS_PER_EDGE[d] * E * (8 * EDGES_PER_CELL[d] + 2)
        f += E * (40 * d + 40 * d * 12)
    return dict(bytes=b, flops=f)


# ---------------------------------------------------------------------------
# The same results in 64 bits, by plain torch
# ---------------------------------------------------------------------------
ROOT_TERMS = 6e9  # edges x support vectors up to which the roots are solved here


class _Lattice:
    """Coordinates, domain and key packing of one triangulation."""

    def __init__(self, w, lam):
        d = self.d = w.d
        self.lam = lam
        self.c = (1.0 - 1.0 / math.sqrt(d + 1.0)) / d
        self.o, self.lo, self.hi = (_dev(v) for v in (w.offset, w.lo, w.hi))
        cinv = self.c * math.sqrt(d + 1.0)
        s0, s1 = float((self.lo - self.o).sum()), float((self.hi - self.o).sum())
        self.y0 = [int(math.floor((float(self.lo[k] - self.o[k]) + cinv * s0) / lam)) - 4
                   for k in range(d)]
        self.span = [int(math.ceil((float(self.hi[k] - self.o[k]) + cinv * s1) / lam)) + 5 - self.y0[k]
                     for k in range(d)]
        self.s0, self.sspan = sum(self.y0), sum(self.span)
        self.cinv = cinv

    def x(self, y):
        cs = self.c * y.sum(1, keepdim=True).double()
        return self.lam * (y.double() - cs) + self.o

    def inside(self, y):
        x = self.x(y)
        return ((x >= self.lo) & (x <= self.hi)).all(1)

    def key(self, y):
        k = y.sum(1) - self.s0
        for i in range(self.d - 2, -1, -1):
            k = k * self.span[i] + (y[:, i] - self.y0[i])
        return k

    def unkey(self, k):
        y = torch.empty((k.shape[0], self.d), dtype=torch.int64, device=k.device)
        for i in range(self.d - 1):
            y[:, i] = k % self.span[i] + self.y0[i]
            k = torch.div(k, self.span[i], rounding_mode="floor")
        y[:, self.d - 1] = k + self.s0 - y[:, :self.d - 1].sum(1)
        return y

    def step(self, mask):
        """e(mask) for a tensor of masks."""
        return torch.stack([(mask >> i) & 1 for i in range(self.d)], 1)


def _found(keys, table):
    """(whether each key is in the sorted table, its place)."""
    if table.shape[0] == 0:
        return torch.zeros_like(keys, dtype=torch.bool), torch.zeros_like(keys)
    at = torch.searchsorted(table, keys).clamp_(max=table.shape[0] - 1)
    return table[at] == keys, at


class _Values:
    """f at lattice vertices, each computed once."""

    def __init__(self, lat, w):
        self.lat, self.w = lat, w
        self.k = torch.empty(0, dtype=torch.int64, device="cuda")
        self.v = torch.empty(0, dtype=torch.float64, device="cuda")

    def at(self, keys):
        uniq = torch.unique(keys)
        new = uniq[~_found(uniq, self.k)[0]]
        if new.shape[0]:
            w = self.w
            f = _f(self.lat.x(self.lat.unkey(new)), w.sv, w.alpha, w.gamma, w.b)
            k = torch.cat([self.k, new])
            order = torch.argsort(k)
            self.k, self.v = k[order], torch.cat([self.v, f])[order]
        return self.v[_found(keys, self.k)[1]]


def _partners(lat, val, edges):
    """The other crossing edge of every 2-simplex coface of the edges (keys)."""
    d, full = lat.d, (1 << lat.d) - 1
    y, S = lat.unkey(edges >> d), edges & full
    y2 = y + lat.step(S)
    f0, f1 = val.at(lat.key(y)), val.at(lat.key(y2))
    got = []
    for M in range(1, full + 1):
        e = lat.step(torch.full((1,), M, dtype=torch.int64, device="cuda"))
        sub, dis = ((M & ~S) == 0) & (S != M), (M & S) == 0
        for pick, base, sign in ((sub, y, 1), (dis, y2, 1), (dis, y, -1)):
            v = base[pick] + sign * e
            ok = lat.inside(v)
            at = pick.nonzero()[:, 0][ok]
            got.append((M, sign if base is y else 2, at, v[ok]))
    wk = lat.key(torch.cat([g[3] for g in got]))
    fw = val.at(wk)
    out, a = [], 0
    for M, how, at, v in got:
        n = at.shape[0]
        k, f = wk[a:a + n], fw[a:a + n]
        a += n
        s, ky, ky2 = S[at], lat.key(y[at]), lat.key(y2[at])
        cross0 = (f >= 0) != (f0[at] >= 0)
        m = torch.full_like(s, M)
        if how == 1:      # y + e(M), M in S
            b, q = torch.where(cross0, ky, k), torch.where(cross0, m, s & ~m)
        elif how == 2:    # y + e(S) + e(M), M disjoint from S
            b, q = torch.where(cross0, ky, ky2), torch.where(cross0, s | m, m)
        else:             # y - e(M)
            b, q = k, torch.where(cross0, m, m | s)
        out.append((b << d) | q)
    return torch.unique(torch.cat(out))


def _seed_edges(lat, val, w):
    d = lat.d
    x = w.seeds
    s = (x - lat.o).sum(1, keepdim=True)
    yp = ((x - lat.o) + lat.cinv * s) / lat.lam
    y = yp.floor().long()
    perm = torch.sort(yp - y, dim=1, descending=True, stable=True)[1]
    verts = [y]
    for j in range(d):
        v = verts[-1].clone()
        v.scatter_add_(1, perm[:, j:j + 1], torch.ones_like(perm[:, :1]))
        verts.append(v)
    out = []
    for i in range(d):
        for j in range(i + 1, d + 1):
            ok = lat.inside(verts[i]) & lat.inside(verts[j])
            a, b = verts[i][ok], verts[j][ok]
            if a.shape[0] == 0:
                continue
            mask = ((b - a) << torch.arange(d, device="cuda")).sum(1)
            cross = (val.at(lat.key(a)) >= 0) != (val.at(lat.key(b)) >= 0)
            out.append(((lat.key(a) << d) | mask)[cross])
    if not out:
        return torch.empty(0, dtype=torch.int64, device="cuda")
    return torch.unique(torch.cat(out))


def _solve(w, x1, dx):
    """t with f(x1 + t dx) = 0, by Newton steps kept in a bracket."""
    n = x1.shape[0]
    t = torch.empty(n, dtype=torch.float64, device="cuda")
    step = max(1, int(2e7) // w.sv.shape[0])
    for a in range(0, n, step):
        p, u = x1[a:a + step], dx[a:a + step]

        def g(q):
            r2 = torch.zeros((p.shape[0], w.sv.shape[0]), dtype=torch.float64, device="cuda")
            proj = torch.zeros_like(r2)
            for k in range(p.shape[1]):
                e = (p[:, k] + q * u[:, k])[:, None] - w.sv[None, :, k]
                r2 += e * e
                proj += e * u[:, k, None]
            e = r2.mul_(-w.gamma).exp_().mul_(w.alpha)
            return e.sum(1) + w.b, -2.0 * w.gamma * (e * proj).sum(1)

        lo, hi = torch.zeros(p.shape[0], dtype=torch.float64, device="cuda"), \
            torch.ones(p.shape[0], dtype=torch.float64, device="cuda")
        f0, f1 = g(lo)[0], g(hi)[0]
        s0 = f0 >= 0
        q = (f0 / (f0 - f1)).clamp(0.0, 1.0)
        for _ in range(60):
            f, df = g(q)
            same = (f >= 0) == s0
            lo, hi = torch.where(same, q, lo), torch.where(same, hi, q)
            nq = q - f / df
            nq = torch.where((nq > lo) & (nq < hi), nq, 0.5 * (lo + hi))
            moved = float((nq - q).abs().max())
            q = nq
            if moved <= 1e-15:
                break
        t[a:a + step] = q
    return t


def _edges(lat, val, w, keys):
    """f, t and the points of the edges (sorted keys); t and the points None
    where they would take long."""
    d = lat.d
    y = lat.unkey(keys >> d)
    y2 = y + lat.step(keys & ((1 << d) - 1))
    f = torch.stack([val.at(lat.key(y)), val.at(lat.key(y2))], 1)
    if keys.shape[0] * w.sv.shape[0] > ROOT_TERMS:
        return dict(edge_f=f, edge_t=None, points=None)
    x1 = lat.x(y)
    dx = lat.x(y2) - x1
    t = _solve(w, x1, dx)
    return dict(edge_f=f, edge_t=t, points=x1 + t[:, None] * dx)


def _traced(w, lam):
    lat = _Lattice(w, lam)
    val = _Values(lat, w)
    front = _seed_edges(lat, val, w)
    seen, last = [front], front[:0]
    while front.shape[0]:
        new = _partners(lat, val, front)
        new = new[~_found(new, front)[0]]
        new = new[~_found(new, last)[0]]
        last, front = front, new
        seen.append(front)
    return lat, val, torch.sort(torch.cat(seen))[0]


def _subdivided(w, lam, k):
    """The crossing edges of scale lam inside the crossing n-simplices of
    scale k lam, as sorted keys."""
    d = w.d
    clat, cval, ce = _traced(w, k * lam)
    # the crossing n-simplices: orderings of each traced edge's two parts
    cells = []
    masks = ce & ((1 << d) - 1)
    for S in torch.unique(masks).tolist():
        y = clat.unkey(ce[masks == S] >> d)
        p1, p2 = [i for i in range(d) if (S >> i) & 1], [i for i in range(d) if not (S >> i) & 1] + [d]
        for a in itertools.permutations(p1):
            for b in itertools.permutations(p2):
                at = b.index(d)
                z = y.clone()
                for i in b[at:]:
                    if i < d:
                        z[:, i] -= 1
                pi = list(b[at + 1:]) + list(a) + list(b[:at])
                code = 0
                for i in pi:
                    code = code * 8 + i
                cells.append((clat.key(z) << (3 * d)) | code)
    cells = torch.unique(torch.cat(cells))
    z = clat.unkey(cells >> (3 * d))
    pi = torch.stack([(cells >> (3 * (d - 1 - j))) & 7 for j in range(d)], 1)
    lat = _Lattice(w, lam)
    val = _Values(lat, w)
    out = []
    local = [v for v in itertools.product(range(k + 1), repeat=d)
             if all(v[i] >= v[i + 1] for i in range(d - 1))]
    for v in local:
        y = k * z
        y.scatter_add_(1, pi, torch.tensor(v, device="cuda").expand_as(pi))
        for M in range(1, 1 << d):
            v2 = [v[i] + ((M >> i) & 1) for i in range(d)]
            if v2[0] > k or any(v2[i] < v2[i + 1] for i in range(d - 1)):
                continue
            bits = torch.tensor([(M >> i) & 1 for i in range(d)], device="cuda").expand_as(pi)
            m = (bits << pi).sum(1)
            out.append(torch.unique((lat.key(y) << d) | m))
    keys = torch.unique(torch.cat(out))
    y = lat.unkey(keys >> d)
    y2 = y + lat.step(keys & ((1 << d) - 1))
    ok = lat.inside(y) & lat.inside(y2)
    keys, y, y2 = keys[ok], y[ok], y2[ok]
    cross = (val.at(lat.key(y)) >= 0) != (val.at(lat.key(y2)) >= 0)
    return lat, val, keys[cross]


def _distance(kind, pose, dims, a, b):
    """Exact distance from the segments a -> b ([n, 3]) to one obstacle: the
    squared distance is convex along the segment, so its slope is bisected."""
    R, t = pose[:9].reshape(3, 3), pose[9:]
    a, b = (a - t) @ R, (b - t) @ R
    u = b - a
    if kind == W.SPHERE:
        uu = (u * u).sum(1)
        q = torch.where(uu > 0, (-(a * u).sum(1) / uu.clamp(min=1e-300)).clamp(0, 1),
                        torch.zeros_like(uu))
        return ((a + q[:, None] * u).norm(dim=1) - dims[0]).clamp(min=0)
    point = not bool(u.any())
    lo, hi = torch.zeros_like(a[:, 0]), torch.ones_like(a[:, 0])

    def parts(q):
        p = a + q[:, None] * u
        if kind == W.BOX:
            e = (p.abs() - dims / 2).clamp(min=0)
            return e, (e * p.sign() * u).sum(1)
        rho = p[:, :2].norm(dim=1)
        e0, e1 = (rho - dims[0]).clamp(min=0), (p[:, 2].abs() - dims[1] / 2).clamp(min=0)
        slope = e0 * (p[:, :2] * u[:, :2]).sum(1) / rho.clamp(min=1e-300) + e1 * p[:, 2].sign() * u[:, 2]
        return torch.stack([e0, e1], 1), slope

    for _ in range(0 if point else 54):
        q = 0.5 * (lo + hi)
        right = parts(q)[1] > 0
        hi, lo = torch.where(right, q, hi), torch.where(right, lo, q)
    best = parts(0.5 * (lo + hi))[0].norm(dim=1)
    for q in (torch.zeros_like(lo), torch.ones_like(lo)):
        best = torch.minimum(best, parts(q)[0].norm(dim=1))
    return best


def _margin(dh, radius, types, pose, dims, points, spheres=None):
    out = []
    for q in points.split(1 << 19):
        n, d = q.shape
        T = torch.eye(4, dtype=torch.float64, device="cuda").repeat(n, 1, 1)
        frames = [T]
        for i in range(d):
            th, dd, aa, al = dh[i]
            c, s = torch.cos(q[:, i] + th), torch.sin(q[:, i] + th)
            ca, sa = torch.cos(al), torch.sin(al)
            A = torch.zeros((n, 4, 4), dtype=torch.float64, device="cuda")
            A[:, 0, 0], A[:, 0, 1], A[:, 0, 2], A[:, 0, 3] = c, -s * ca, s * sa, aa * c
            A[:, 1, 0], A[:, 1, 1], A[:, 1, 2], A[:, 1, 3] = s, c * ca, -c * sa, aa * s
            A[:, 2, 1], A[:, 2, 2], A[:, 2, 3], A[:, 3, 3] = sa, ca, dd, 1.0
            frames.append(frames[-1] @ A)
        el = [(frames[i][:, :3, 3], frames[i + 1][:, :3, 3], radius[i]) for i in range(d)]
        if spheres is not None:
            for link, centre, r in zip(spheres[0].tolist(), spheres[1], spheres[2]):
                p = frames[link + 1][:, :3, :3] @ centre + frames[link + 1][:, :3, 3]
                el.append((p, p, r))
        best = torch.full((n,), -math.inf, dtype=torch.float64, device="cuda")
        for a, b, r in el:
            for j, kind in enumerate(types.tolist()):
                best = torch.maximum(best, r - _distance(kind, pose[j], dims[j], a, b))
        out.append(best)
    return torch.cat(out)


def exact(case, seed):
    kind = case["kind"]
    if kind == "certify":
        q = _sampled_scene(case, seed)
        return dict(margin=_margin(q["dh"], q["radius"], q["types"], q["pose"], q["dims"],
                                   q["points"], q["spheres"]))
    if kind in ("batch", "served"):
        got = []
        for w in _shells(case, seed):
            lat, val, keys = _traced(w, w.lam)
            got.append(_edges(lat, val, w, keys))
        return {k: None if any(e[k] is None for e in got) else
                torch.cat([e[k].reshape(-1) for e in got]) for k in ("edge_f", "edge_t", "points")}
    w = _problem(case, seed)
    if kind == "eval":
        return _f(_points(case, w, seed), w.sv, w.alpha, w.gamma, w.b)
    E0, lam0 = EDGES_REF[case["d"]]
    if E0 * (lam0 / case["lam"]) ** (case["d"] - 1) * case["n_sv"] > 4 * ROOT_TERMS:
        return None
    lat, val, keys = _subdivided(w, w.lam, case["k"]) if kind == "subdiv" else _traced(w, w.lam)
    out = _edges(lat, val, w, keys)
    if kind == "proof" and out["points"] is not None and keys.shape[0]:
        out["margin"] = _margin(w.dh, w.radius, w.obs_type, w.obs_pose, w.obs_dims, out["points"])
    return out
