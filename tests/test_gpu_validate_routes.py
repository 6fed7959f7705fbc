"""GPU: the verdict kernel's routes (an edge per warp, an edge per block; with
and without a distance field) against the unculled clearance kernel: an edge is
valid exactly when its minimum clearance is at least the margin.  Edges within
2e-5 m of the margin, where FP32 rounding of a clearance decides, are left out;
both kernels place the spheres with the same arithmetic, so few are."""
import dataclasses

import numpy as np
import pytest
import torch

from paper_2609_30644_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def mp():
    assert torch.cuda.is_available()
    import paper_2609_30644_gb300 as m
    return m


def _far(o, d):
    o = o.copy()
    o[:, :3] += np.float32(d)
    return o


def _scene(kind):
    table = synth.table_pair_scene(0)
    none = dict(obs_spheres=table.obs_spheres[:0], obs_cuboids=table.obs_cuboids[:0])
    if kind == "planar":
        return synth.planar_pair_scene(1)
    if kind == "table":
        return table
    if kind.startswith("batched"):
        return synth.batched_scene(int(kind[7:]))
    if kind == "one_arm":
        return dataclasses.replace(table, robots=table.robots[:1])
    if kind == "no_obstacles":      # close bases: the arms' pairs decide
        b = table.robots[1].base.copy()
        b[7] = -0.25
        return dataclasses.replace(table, robots=[table.robots[0],
                                                  dataclasses.replace(table.robots[1], base=b)], **none)
    if kind == "out_of_reach":      # every obstacle beyond every link
        return dataclasses.replace(table, obs_spheres=_far(table.obs_spheres, 50.0),
                                   obs_cuboids=_far(table.obs_cuboids, -1e6))
    if kind == "one_far":           # a scattered scene: the field covers the reach only
        s = table.obs_spheres.copy()
        s[0, :3] = 1e5
        return dataclasses.replace(table, obs_spheres=s)
    if kind == "offset":            # coordinates too large for the field's index arithmetic
        robots = []
        for r in table.robots:
            b = r.base.copy()
            b[[3, 7, 11]] += np.float32(65536.0)
            robots.append(dataclasses.replace(r, base=b))
        return dataclasses.replace(table, robots=robots, obs_spheres=_far(table.obs_spheres, 65536.0),
                                   obs_cuboids=_far(table.obs_cuboids, 65536.0))
    if kind == "bare_links":        # links and a whole robot without spheres
        r0, r1 = table.robots
        keep = np.isin(r0.sphere_link, [1, 4])
        a = dataclasses.replace(r0, sphere_link=r0.sphere_link[keep], sphere_xyzr=r0.sphere_xyzr[keep])
        b = dataclasses.replace(r1, sphere_link=r1.sphere_link[:0], sphere_xyzr=r1.sphere_xyzr[:0])
        return dataclasses.replace(table, robots=[b, a, r1])
    if kind == "big_spheres":       # one coarse radius far above the others
        r0, r1 = table.robots
        x = r0.sphere_xyzr.copy()
        x[-1, 3] = 0.6
        return dataclasses.replace(table, robots=[dataclasses.replace(r0, sphere_xyzr=x), r1])
    raise ValueError(kind)


@pytest.mark.parametrize("kind,n,self_collision", [
    ("planar", 1, False), ("planar", 300, False), ("planar", 5000, True), ("table", 500, False),
    ("table", 6000, False), ("one_arm", 700, False), ("one_arm", 7000, False),
    ("no_obstacles", 400, False), ("no_obstacles", 6000, False), ("out_of_reach", 2000, False),
    ("one_far", 2000, False), ("offset", 500, False), ("bare_links", 3000, False),
    ("big_spheres", 3000, False), ("batched10", 200, False), ("batched10", 1500, False),
    ("batched9", 800, True)])
@pytest.mark.parametrize("margin", [1e-4, 0.02])
def test_verdict_is_clearance_at_margin(mp, kind, n, self_collision, margin):
    scene = _scene(kind)
    qa, qb = synth.candidate_edges(scene, n, seed=n, step_hi=2.0)
    if n > 8:
        qb[:, 3] = qa[:, 3]          # a single configuration
        qb[0, 5] = np.nan            # invalid unchecked
    qa, qb = torch.from_numpy(qa).cuda(), torch.from_numpy(qb).cuda()
    with mp.Problem(scene, margin=margin, self_collision=self_collision) as p:
        clear = mp.edge_clearance(p, qa, qb).cpu().numpy()
        length = torch.empty(n, device="cuda")
        points = torch.empty(n, dtype=torch.int32, device="cuda")
        # (at coordinates of 65,536 m FP32 resolves 8 mm)
        band = 2e-5 if kind != "offset" else 0.05
        decided = ~(np.abs(clear - np.float32(margin)) < band)
        for order in (0, 1):
            for warps in (4, 1):     # one warp per block: no group launch
                mp.set_launch(p, warps, order)
                for regs in (0, 1):
                    mp.set_launch(p, warps, order, 0, regs)
                    v = mp.validate_edges(p, qa, qb, length=length, npoints=points).cpu().numpy()
                    np.testing.assert_array_equal(v[decided], (clear >= margin)[decided])
        if n > 8:
            assert v[5] == 0
        if kind in ("table", "no_obstacles") and n > 8:
            assert 0.05 < v.mean() < 0.95     # both verdicts are exercised
        d = (qb - qa).double().norm(dim=0)
        ok = torch.isfinite(d)
        torch.testing.assert_close(length.double()[ok], d[ok], rtol=1e-6, atol=1e-7)


@pytest.mark.parametrize("kind,n,chunks", [
    ("planar", 20000, (300, 1500, 4000)), ("table", 30000, (700, 1900, 2300, 9000))])
def test_verdicts_do_not_depend_on_the_batch(mp, kind, n, chunks):
    """An edge's verdict is the same in a batch that gives each warp many edges,
    in one whose idle warps help and with a block to an edge."""
    scene = _scene(kind)
    qa, qb = synth.candidate_edges(scene, n, seed=5, step_hi=2.0)
    qa, qb = torch.from_numpy(qa).cuda(), torch.from_numpy(qb).cuda()
    with mp.Problem(scene, margin=1e-4) as p:
        whole = mp.validate_edges(p, qa, qb).cpu()
        assert 0 < int(whole.sum()) < n
        for c in chunks:
            for e0 in range(0, 3 * c, c):
                a, b = (x[:, e0:e0 + c].contiguous() for x in (qa, qb))
                assert torch.equal(mp.validate_edges(p, a, b).cpu(), whole[e0:e0 + c])
