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
