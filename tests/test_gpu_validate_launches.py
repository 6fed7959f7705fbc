"""GPU: every launch form of the verdict kernel gives an edge the same verdict.
The reference is an edge per warp and one warp per block, which shares nothing
between warps."""
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


# edges of up to some 80 tiles, an edge to a block: the warps that share an edge
# leave it on whichever warp's tile collides
@pytest.mark.parametrize("make,n", [(synth.planar_pair_scene, 1), (synth.planar_pair_scene, 300),
                                    (synth.table_pair_scene, 7), (synth.table_pair_scene, 500)])
@pytest.mark.parametrize("order", [0, 1])
def test_block_per_edge_of_many_tiles(mp, make, n, order):
    scene = make(0)
    qa, qb = synth.candidate_edges(scene, n, seed=n, step_lo=0.5, step_hi=5.0)
    if n > 8:
        qb[0, 5] = np.nan            # invalid unchecked
    qa, qb = torch.from_numpy(qa).cuda(), torch.from_numpy(qb).cuda()
    with mp.Problem(scene, resolution=0.002, margin=1e-4) as p:
        mp.set_launch(p, 1, order)
        want = mp.validate_edges(p, qa, qb).cpu()
        if n > 8:
            assert want[5] == 0 and 0 < int(want.sum()) < n
        for warps in (2, 4):
            mp.set_launch(p, warps, order)
            for _ in range(3):
                assert torch.equal(mp.validate_edges(p, qa, qb).cpu(), want)


def _one_arm_with_cuboids(n):
    """A 7-joint arm among n small boxes on a shell it can reach (tables of
    80 bytes a box: more than 48 KB of shared memory a block)."""
    table = synth.table_pair_scene(0)
    rng = np.random.default_rng(n)
    arm = table.robots[0]
    c = rng.standard_normal((n, 3))
    c *= rng.uniform(0.75, 1.3, (n, 1)) / np.linalg.norm(c, axis=1, keepdims=True)
    box = np.zeros((n, 15), np.float32)
    box[:, :3] = c + arm.base.reshape(3, 4)[:, 3]
    box[:, 3:6] = rng.uniform(0.005, 0.02, (n, 3))
    box[:, 6:] = np.eye(3, dtype=np.float32).ravel()
    return synth.Scene([arm], table.obs_spheres[:0], box)


# batches beyond the block-per-edge and the shared forms, with more shared memory
# a block than a kernel has by default, in both register budgets
@pytest.mark.parametrize("make,n", [(lambda: synth.batched_scene(10), 16384),
                                    (lambda: synth.batched_scene(0), 16384),
                                    (lambda: _one_arm_with_cuboids(700), 5000),
                                    (lambda: _one_arm_with_cuboids(1024), 1400)])
@pytest.mark.parametrize("regs", [0, 1])
def test_large_tables_in_large_batches(mp, make, n, regs):
    scene = make()
    qa, qb = synth.candidate_edges(scene, n, seed=3)
    qa, qb = torch.from_numpy(qa).cuda(), torch.from_numpy(qb).cuda()
    with mp.Problem(scene, margin=1e-4) as p:
        parts = [mp.validate_edges(p, qa[:, i:i + 512].contiguous(), qb[:, i:i + 512].contiguous())
                 for i in range(0, n, 512)]
        want = torch.cat(parts).cpu()
        assert 0 < int(want.sum()) < n
        for warps in (4, 1):
            mp.set_launch(p, warps, 0, 0, regs)
            assert torch.equal(mp.validate_edges(p, qa, qb).cpu(), want)


def test_autotune_large_tables(mp):
    mp.autotune_cache_clear()
    scene = _one_arm_with_cuboids(700)
    qa, qb = (torch.from_numpy(a).cuda() for a in synth.candidate_edges(scene, 5000, seed=4))
    with mp.Problem(scene, margin=1e-4) as p:
        want = mp.validate_edges(p, qa, qb)
        assert mp.autotune(p, qa, qb)[0] in (1, 2, 4)
        assert torch.equal(mp.validate_edges(p, qa, qb), want)
    mp.autotune_cache_clear()
