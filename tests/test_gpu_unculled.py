"""GPU: verdicts and clearances against a check that culls nothing.  The verdict
and the clearance kernels share their coarse spheres, tile bounds and slacks, so
that agreeing with each other does not show that these enclose what they
replace; here both are compared with the FP64 oracle, which measures every pair,
in the scenes that stress the bounds.  Each batch holds a few distinct edges
many times over, so that every launch form decides them.

Tolerances: clearances |gpu - oracle| <= 1e-5 (1 + |oracle|), verdicts exact
outside a 1e-4 m band around the margin.  At coordinates of 65,536 m half a unit
in the last place is 2^-8 m: a 7-joint chain adds at most 14 link offsets, and a
sphere centre and a distance one rounding each, along three axes."""
import numpy as np
import pytest
import torch

from paper_2609_30644_gb300 import synth
from test_gpu_validate_routes import _scene

pytestmark = pytest.mark.gpu

OFFSET_TOL = 16 * 2.0 ** -8 * 3.0 ** 0.5


@pytest.fixture(scope="module")
def mp():
    assert torch.cuda.is_available()
    import paper_2609_30644_gb300 as m
    return m


@pytest.mark.parametrize("kind,n,self_collision,step", [
    ("planar", 200, False, 2.0), ("planar", 100, True, 2.0), ("one_arm", 120, False, 2.0),
    ("no_obstacles", 80, False, 2.0), ("out_of_reach", 60, False, 1.0), ("one_far", 80, False, 1.0),
    ("offset", 60, False, 1.0), ("bare_links", 100, False, 1.0), ("big_spheres", 100, False, 1.0),
    ("batched10", 150, False, 0.2), ("batched9", 30, True, 0.2)])
@pytest.mark.parametrize("margin", [1e-4, 0.02])
def test_against_all_pairs(mp, orc, kind, n, self_collision, step, margin):
    scene = _scene(kind)
    qa, qb = synth.candidate_edges(scene, n, seed=71, step_lo=0.02, step_hi=step)
    ref = orc.OracleScene(scene, self_collision=self_collision).validate_edges(
        qa, qb, 0.02, margin, early_exit=False)
    want, tol = ref["min_clear"], 1e-5 * (1 + np.abs(ref["min_clear"]))
    band = 1e-4
    if kind == "offset":
        tol = band = OFFSET_TOL
    decided = np.abs(want - margin) > band
    assert decided.sum() >= 8
    a, b = torch.from_numpy(qa).cuda(), torch.from_numpy(qb).cuda()
    with mp.Problem(scene, margin=margin, self_collision=self_collision) as p:
        clear = mp.edge_clearance(p, a, b).cpu().numpy().astype(np.float64)
        assert (np.abs(clear - want) <= tol).all(), np.abs(clear - want).max()
        # a block to an edge, an edge to a warp with and without shared tiles
        for total in (n, 6000, 30000):
            k = -(-total // n)
            v = mp.validate_edges(p, a.repeat(1, k), b.repeat(1, k)).view(k, n).cpu().numpy()
            assert (v == v[0]).all()
            np.testing.assert_array_equal(v[0][decided], ref["valid"][decided])
