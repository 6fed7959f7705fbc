"""GPU: the persistent launch runs a ROADMAP round's phases over all robots at
once; it has to give what the stepped form gives, round for round."""
import numpy as np
import pytest

from paper_2609_30644_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def mp():
    import torch
    assert torch.cuda.is_available()
    import paper_2609_30644_gb300 as m
    return m


def _free_pair(mp, scene, seed):
    import torch
    q = synth.uniform_configs(scene, 4096, synth.rng_for(6, seed))
    with mp.Problem(scene, margin=2e-3) as p:
        qd = torch.from_numpy(q).cuda()
        free = np.nonzero(mp.validate_edges(p, qd, qd).cpu().numpy())[0]
    return q[:, free[0]].copy(), q[:, free[1]].copy()


# new vertices per round at the edges of the 64-vertex link tile (the first
# round gathers two more), one vertex a round, and rounds that pass the shared
# tables' 16,384 vertices
@pytest.mark.parametrize("idx,per_round,steps", [(8, 62, 10), (8, 63, 10), (8, 200, 8), (5, 1, 8),
                                                 (9, 4096, 7)])
def test_persistent_equals_stepped(mp, idx, per_round, steps):
    scene = synth.batched_scene(idx)
    qs, qg = _free_pair(mp, scene, idx)
    got = []
    for form in (mp.BATCH_PERSISTENT, mp.BATCH_STEPPED):
        with mp.Problem(scene, resolution=0.02, margin=1e-4, delta=2.5, n_per_round=per_round,
                        tree_cap=1 << 14, roadmap_cap=1 << 15, max_iters=256, seed=idx,
                        start=qs, goal=qg) as p:
            mp.plan_batch([p], 60.0, max_steps=steps, form=form)
            path, cost = mp.plan_result(p)
            _, costs, iters = mp.plan_trace(p)
            got.append((path, cost, costs, iters))
    a, b = got
    assert a[3] == b[3] and a[1] == b[1]
    np.testing.assert_array_equal(a[2], b[2])
    if a[0] is not None:
        np.testing.assert_array_equal(a[0], b[0])
