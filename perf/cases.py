"""Performance cases of the motion-validation library: the calls that a planner or a
planning service built on it makes, through the public binding, from one search
step's 256 edges up to full batches, with every entry point of the hot path.

Kinds (a case's "kind"):
  validate   composite-edge validation of n candidate edges
  clearance  minimum signed clearance of n edges (or of n single configurations)
  fk         sphere centres of n configurations
  nearest    cost-filtered NEAREST of q queries over a tree of n vertices
  neighbors  radius NEIGHBORS of q queries over n roadmap vertices
  path_cost  cost of a path of n vertices
  plan       a batch of planning requests, from their scenes to their paths

Inputs are synthetic (the generators of the package) and depend on the seed.
"""
import math

import numpy as np
import torch

import paper_2609_30644_gb300 as mp
from paper_2609_30644_gb300 import synth

RES = 0.02          # edge resolution (rad)
MARGIN = 1e-4       # the planner's contact margin (m)
PLAN_DELTA = 2.5    # roadmap connection radius of 7-DOF arms (rad)
ARM_LIMIT = 2.9     # joint limits of the 7-DOF arms (rad)
DEV = "cuda"


# ----------------------------------------------------------------------------
# cases
# ----------------------------------------------------------------------------

def listed():
    return [
        # one search step of the planar pair: 256 extension edges, the smallest call
        dict(name="check_step_planar", kind="validate", scene="planar", n=256, margin=1e-4,
             by_products=False),
        # the benchmark's batch: 65,536 candidate edges of two arms over a table
        dict(name="check_batch_table", kind="validate", scene="table", n=65536, margin=1e-4,
             by_products=False),
        # four arms around a cube with 128 obstacles, a wide margin, a ragged batch
        dict(name="check_grid4", kind="validate", scene="grid4", n=16001, margin=0.02,
             by_products=False),
        # eight arms, 219 obstacles, with the edge lengths and interval counts that
        # a tree insert needs
        dict(name="check_arms8", kind="validate", scene="batched:10", n=4099, margin=1e-4,
             by_products=True),
        # signed clearance along candidate edges (path quality, start/goal choice)
        dict(name="clearance_table", kind="clearance", scene="table", n=1023, still=False),
        # sphere centres of a batch of configurations (visualisation, distance checks)
        dict(name="fk_table", kind="fk", scene="table", n=20001),
        # the benchmark's NEAREST: 65,536 queries over a 16,384-vertex tree
        dict(name="nearest_batch_14d", kind="nearest", dim=14, n=16384, q=65536, filter=0),
        # one search step of four arms over a grown tree: few queries, many vertices
        dict(name="nearest_step_28d", kind="nearest", dim=28, n=100003, q=256, filter=0),
        # a batch over a five-arm (35-DOF) tree
        dict(name="nearest_batch_35d", kind="nearest", dim=35, n=50000, q=8192, filter=0),
        # ROADMAP neighbours of one arm: 1,024 samples against its roadmap
        dict(name="neighbors_roadmap", kind="neighbors", dim=7, n=4096, q=1024, delta=1.2,
             k_max=32),
        # cost of a long path
        dict(name="path_cost_14d", kind="path_cost", dim=14, n=65537),
        # twelve planning requests with 2-8 arms and 16-256 obstacles, each from its
        # scene to its path in one batch
        dict(name="plan_batch", kind="plan", first=1, problems=12, steps=24),
    ]


def _log_int(rng, lo, hi):
    """Integer spread over the logarithm of [lo, hi], odd sizes and powers of two alike."""
    v = int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))
    return min(hi, max(lo, v))


def draw(rng):
    kind = rng.choice(["validate", "validate", "validate", "nearest", "nearest", "nearest",
                       "neighbors", "neighbors", "fk", "path_cost", "clearance", "plan"])
    if kind == "validate":
        scene = rng.choice(["planar", "table", "table", "grid4", "batched:%d" % rng.randrange(24)])
        hi = {"planar": 65536, "table": 65536, "grid4": 32768}.get(scene, 8192)
        return dict(kind=kind, scene=scene, n=_log_int(rng, 64, hi),
                    margin=rng.choice([0.0, 1e-4, 0.02]), by_products=rng.random() < 0.3)
    if kind == "clearance":
        return dict(kind=kind, scene=rng.choice(["planar", "table", "grid4"]),
                    n=_log_int(rng, 64, 1000), still=rng.random() < 0.5)
    if kind == "fk":
        return dict(kind=kind, scene=rng.choice(["planar", "table", "grid4", "batched:8"]),
                    n=_log_int(rng, 64, 65536))
    if kind == "nearest":
        dim = rng.choice([6, 7, 14, 14, 21, 28, 35, 42, 56])
        n = _log_int(rng, 1000, 1000000)
        # as many query-vertex coordinates as the largest listed batch, at most
        most = int(min(65536, 8192 * 50000 * 35 / (n * dim)))
        return dict(kind=kind, dim=dim, n=n, q=_log_int(rng, 64, max(128, most)),
                    filter=int(rng.random() < 0.2))
    if kind == "neighbors":
        dim = rng.choice([3, 7, 7, 7, 14])
        n = _log_int(rng, 100, 32768)
        return dict(kind=kind, dim=dim, n=n, q=_log_int(rng, 64, 8192),
                    delta={3: 0.8, 7: rng.choice([1.2, 2.5]), 14: 4.0}[dim],
                    k_max=rng.choice([16, 32, 64]))
    if kind == "path_cost":
        return dict(kind=kind, dim=rng.choice([6, 7, 14, 28, 56]), n=_log_int(rng, 8, 262144))
    return dict(kind="plan", first=rng.randrange(24), problems=rng.randrange(1, 9),
                steps=rng.randrange(4, 25))


# ----------------------------------------------------------------------------
# inputs
# ----------------------------------------------------------------------------

def _scene(name):
    if name == "planar":
        return synth.planar_pair_scene(0)
    if name == "table":
        return synth.table_pair_scene(0)
    if name == "grid4":
        return synth.grid4_scene(0)
    return synth.batched_scene(int(name.split(":")[1]))


def _gen(seed):
    g = torch.Generator(device=DEV)
    g.manual_seed(int(seed))
    return g


def _box(dim, n, g):
    """float32 [dim, n] uniform in the arms' joint limits."""
    return (torch.rand(dim, n, generator=g, device=DEV) * 2 - 1) * ARM_LIMIT


def _edges(scene, n, seed):
    qa, qb = synth.candidate_edges(scene, n, seed=seed)
    return torch.from_numpy(qa).to(DEV), torch.from_numpy(qb).to(DEV)


def _plan_requests(case, seed):
    """(scene, start, goal) of the batched workload, with start and goal 2 mm
    clear of contact; scenes without such a pair in 8,192 draws are skipped."""
    out, idx = [], case["first"]
    while len(out) < case["problems"]:
        scene = synth.batched_scene(idx)
        q = synth.uniform_configs(scene, 8192, synth.rng_for(6, idx, seed))
        with mp.Problem(scene, resolution=RES, margin=2e-3) as p:
            qd = torch.from_numpy(q).to(DEV)
            ok = mp.validate_edges(p, qd, qd).cpu().numpy()
        free = np.nonzero(ok)[0]
        if len(free) >= 2:
            out.append((scene, q[:, free[0]].copy(), q[:, free[1]].copy(), idx + 1000 * seed))
        idx += 1
    return out


def prepare(case, seed):
    kind = case["kind"]
    if kind == "validate":
        scene = _scene(case["scene"])
        p = mp.Problem(scene, resolution=RES, margin=case["margin"])
        qa, qb = _edges(scene, case["n"], seed)
        return dict(kind=kind, p=p, qa=qa, qb=qb, by_products=case["by_products"])
    if kind == "clearance":
        scene = _scene(case["scene"])
        p = mp.Problem(scene, resolution=RES, margin=MARGIN)
        qa, qb = _edges(scene, case["n"], seed)
        return dict(kind=kind, p=p, qa=qa, qb=qa if case["still"] else qb)
    if kind == "fk":
        scene = _scene(case["scene"])
        p = mp.Problem(scene, resolution=RES, margin=MARGIN)
        qa, _ = _edges(scene, case["n"], seed)
        return dict(kind=kind, p=p, q=qa)
    if kind == "nearest":
        g, dim, n, q = _gen(seed), case["dim"], case["n"], case["q"]
        diag = 2 * ARM_LIMIT * math.sqrt(dim)
        tree = torch.empty(dim + 1, n, device=DEV)
        tree[:dim] = _box(dim, n, g)
        tree[dim] = torch.rand(n, generator=g, device=DEV) * (2 * diag)   # cost-to-come
        tree[dim, 0] = 0.0
        queries = _box(dim, q, g)
        # budgets from near the root's reach to almost the whole tree
        budgets = (0.45 + 1.4 * torch.rand(q, generator=g, device=DEV)) * diag
        return dict(kind=kind, tree=tree, queries=queries, budgets=budgets,
                    filter=case["filter"])
    if kind == "neighbors":
        g = _gen(seed)
        return dict(kind=kind, tree=_box(case["dim"], case["n"], g),
                    queries=_box(case["dim"], case["q"], g), delta=case["delta"],
                    k_max=case["k_max"])
    if kind == "path_cost":
        g = _gen(seed)
        step = torch.randn(case["n"], case["dim"], generator=g, device=DEV) * 0.05
        return dict(kind=kind, path=torch.cumsum(step, dim=0).contiguous())
    return dict(kind=kind, requests=_plan_requests(case, seed), steps=case["steps"])


# ----------------------------------------------------------------------------
# one pass
# ----------------------------------------------------------------------------

def _run_plan(s):
    """A service's batch: problems from their scenes, one planner launch, results out."""
    ps = [mp.Problem(scene, resolution=RES, margin=MARGIN, delta=PLAN_DELTA, n_per_round=64,
                     tree_cap=1 << 15, roadmap_cap=1 << 13, max_iters=4096, seed=sd, start=qs,
                     goal=qg) for scene, qs, qg, sd in s["requests"]]
    status = mp.plan_batch(ps, 100.0, max_steps=s["steps"])
    # paths of up to 512 vertices in up to 56 dimensions, zero-padded to one shape
    costs, paths = np.zeros(len(ps)), np.zeros((len(ps), 512, 56), np.float32)
    for i, p in enumerate(ps):
        path, costs[i] = mp.plan_result(p, path_cap=512)
        if path is not None:
            paths[i, :path.shape[0], :path.shape[1]] = path
        p.close()
    return dict(status=status, cost=costs, path=paths)


def run(s):
    kind = s["kind"]
    if kind == "validate":
        if not s["by_products"]:
            return mp.validate_edges(s["p"], s["qa"], s["qb"])
        n = s["qa"].shape[1]
        length = torch.empty(n, dtype=torch.float32, device=DEV)
        npoints = torch.empty(n, dtype=torch.int32, device=DEV)
        valid = mp.validate_edges(s["p"], s["qa"], s["qb"], length=length, npoints=npoints)
        return [valid, length, npoints]
    if kind == "clearance":
        return mp.edge_clearance(s["p"], s["qa"], s["qb"])
    if kind == "fk":
        return mp.fk(s["p"], s["q"])
    if kind == "nearest":
        return mp.nearest(s["tree"], s["queries"], s["budgets"], filter=s["filter"])
    if kind == "neighbors":
        return mp.neighbors(s["tree"], s["queries"], s["delta"], s["k_max"])
    if kind == "path_cost":
        return mp.path_cost(s["path"])
    return _run_plan(s)


# ----------------------------------------------------------------------------
# what a pass cannot do without
# ----------------------------------------------------------------------------

def _mean_points(scene):
    """Mean checkpoints per candidate edge, from the edge distribution."""
    qa, qb = synth.candidate_edges(scene, 2048, seed=1)
    d = np.sqrt(((qb.astype(float) - qa) ** 2).sum(0))
    return float(np.maximum(1, np.ceil(d / RES)).mean()) + 1


def work(case):
    kind = case["kind"]
    if kind in ("validate", "clearance", "fk"):
        scene = _scene(case["scene"])
        n, D = case["n"], scene.D
        S = sum(r.n_spheres for r in scene.robots)
        if kind == "fk":
            # a joint transform per link, a point transform per sphere
            return dict(bytes=4.0 * n * (D + 3 * S), flops=float(n) * (51 * D + 18 * S))
        points = 1.0 if case.get("still") else _mean_points(scene)
        # every checkpoint of a valid edge needs its chain and its links' bounding
        # centres; about half of the candidate edges are valid, the others need
        # one checkpoint
        per_edge = 0.5 * (points + 1) if kind == "validate" else points
        out = (1 + 8 * bool(case.get("by_products"))) if kind == "validate" else 4
        return dict(bytes=float(n) * (8 * D + out), flops=n * per_edge * D * (51.0 + 18.0))
    if kind == "nearest":
        n, q, dim = case["n"], case["q"], case["dim"]
        # vertices with a cost-to-come below the budget: 0.575 of them on average
        return dict(bytes=4.0 * (dim + 1) * (n + q) + 8.0 * q, flops=0.575 * n * q * 2.0 * dim)
    if kind == "neighbors":
        n, q, dim = case["n"], case["q"], case["dim"]
        return dict(bytes=4.0 * dim * (n + q) + 8.0 * q * (case["k_max"] + 1),
                    flops=3.0 * dim * n * q)
    if kind == "path_cost":
        n, dim = case["n"], case["dim"]
        return dict(bytes=4.0 * n * dim + 8, flops=3.0 * n * dim)
    # plan: every search step checks up to 256 extension edges of about 34
    # points in 7 K dimensions (K = 5 on average)
    edges = case["problems"] * case["steps"] * 256.0
    return dict(bytes=edges * 2 * 35 * 4, flops=edges * 0.5 * 34 * 35 * 69.0)


# ----------------------------------------------------------------------------
# 64-bit values of the computed outputs
# ----------------------------------------------------------------------------

def _f64(a):
    return torch.as_tensor(np.asarray(a, dtype=np.float64), device=DEV)


def _fk64(scene, q):
    """Sphere centres [S, n, 3] of configurations q [D, n] (float64)."""
    n, off, out = q.shape[1], 0, []
    for r in scene.robots:
        base = _f64(np.asarray(r.base, np.float32).reshape(3, 4))
        R = base[:, :3].expand(n, 3, 3)
        t = base[:, 3].expand(n, 3)
        dh, xyzr, link = _f64(r.dh), _f64(r.sphere_xyzr), torch.as_tensor(np.asarray(r.sphere_link))
        for j in range(r.dof):
            th = q[off + j] + dh[j, 3]
            c, s = torch.cos(th), torch.sin(th)
            z, one = torch.zeros_like(c), torch.ones_like(c)
            Rz = torch.stack([c, -s, z, s, c, z, z, z, one], dim=1).reshape(n, 3, 3)
            F = R @ Rz
            sel = torch.nonzero(link == j).ravel().tolist()
            if sel:
                out.append((torch.einsum("nij,sj->sni", F, xyzr[sel, :3]) + t))
            t = t + F[:, :, 2] * dh[j, 2] + F[:, :, 0] * dh[j, 0]
            ca, sa = torch.cos(dh[j, 1]), torch.sin(dh[j, 1])
            R = torch.stack([F[:, :, 0], F[:, :, 1] * ca + F[:, :, 2] * sa,
                             F[:, :, 2] * ca - F[:, :, 1] * sa], dim=2)
        off += r.dof
    return torch.cat(out, dim=0)


def _clear64(scene, q):
    """Minimum signed clearance of configurations q [D, n] (float64), [n]."""
    X = _fk64(scene, q)                                            # [S, n, 3]
    rad = _f64(np.concatenate([r.sphere_xyzr[:, 3] for r in scene.robots]))
    who = np.concatenate([[k] * r.n_spheres for k, r in enumerate(scene.robots)])
    best = torch.full((q.shape[1],), float("inf"), dtype=torch.float64, device=DEV)
    osph, ocub = _f64(scene.obs_spheres), _f64(scene.obs_cuboids)
    for i in range(len(osph)):
        d = (X - osph[i, :3]).norm(dim=2) - rad[:, None] - osph[i, 3]
        best = torch.minimum(best, d.amin(0))
    for i in range(len(ocub)):
        R = ocub[i, 6:].reshape(3, 3)
        u = (((X - ocub[i, :3]) @ R).abs() - ocub[i, 3:6]).clamp(min=0)
        best = torch.minimum(best, (u.norm(dim=2) - rad[:, None]).amin(0))
    for s in range(1, len(rad)):
        o = torch.as_tensor(np.nonzero(who[:s] != who[s])[0], device=DEV)
        if len(o):
            d = (X[o] - X[s]).norm(dim=2) - rad[o][:, None] - rad[s]
            best = torch.minimum(best, d.amin(0))
    return best


def exact(case, seed):
    kind = case["kind"]
    if kind == "validate" and case["by_products"]:
        scene = _scene(case["scene"])
        qa, qb = synth.candidate_edges(scene, case["n"], seed=seed)
        return [None, np.sqrt(((qb.astype(np.float64) - qa) ** 2).sum(0)), None]
    if kind == "fk":
        scene = _scene(case["scene"])
        qa, _ = synth.candidate_edges(scene, case["n"], seed=seed)
        return _fk64(scene, _f64(qa)).permute(2, 0, 1).contiguous()
    if kind == "clearance":
        scene, n = _scene(case["scene"]), case["n"]
        qa, qb = synth.candidate_edges(scene, n, seed=seed)
        if case["still"]:
            qb = qa
        a, d = _f64(qa), _f64(qb) - _f64(qa)
        steps = torch.ceil(d.norm(dim=0) / RES).clamp(min=1).long()
        best = torch.full((n,), float("inf"), dtype=torch.float64, device=DEV)
        for k in range(int(steps.max()) + 1):
            on = torch.nonzero(steps >= k).ravel()
            f = k / steps[on].double()
            best[on] = torch.minimum(best[on], _clear64(scene, a[:, on] + f * d[:, on]))
        return best
    if kind == "path_cost":
        path = prepare(case, seed)["path"].double()
        return (path[1:] - path[:-1]).norm(dim=1).sum().reshape(1)
    return None
