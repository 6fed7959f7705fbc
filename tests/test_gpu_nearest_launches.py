"""GPU: the slice waves of the budget-ordered NEAREST (its autotuner's knob)
change the launch, never an index, at sizes that take that path with either
filter.  The reference is the scan, through batches too small for any other
route."""
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


@pytest.mark.parametrize("D,n,Q,filt", [(14, 17001, 3001, 0), (14, 17001, 3001, 1),
                                        (35, 9001, 2049, 0), (28, 9001, 2600, 1)])
def test_slice_waves(mp, tmp_path, D, n, Q, filt):
    lo, hi = -2.9 * np.ones(D), 2.9 * np.ones(D)
    diag = float(np.sqrt(D) * 5.8)
    tree = torch.from_numpy(synth.random_tree_fast(D, n, lo, hi, seed=D)).cuda()
    qs, cs = synth.nn_queries(D, Q, lo, hi, seed=D + 1, budget_lo=0.3 * diag, budget_hi=1.9 * diag)
    q, c = torch.from_numpy(qs).cuda(), torch.from_numpy(cs).cuda()
    want = torch.cat([mp.nearest(tree, q[:, i:i + 64].contiguous(), c[i:i + 64].contiguous())
                      for i in range(0, Q, 64)])
    assert 0 < int((want >= 0).sum())
    # the ordered path skips pairs, the scan none
    assert mp.nearest_work(tree, q, c) < n * Q
    mp.autotune_cache_clear()
    got, waves, ms = mp.nearest_autotune(tree, q, c, filter=filt)
    assert waves in (2, 4, 8) and ms > 0 and torch.equal(got, want)
    path = tmp_path / "tuned.txt"
    mp.autotune_cache_save(str(path))
    key = [l.split(" = ")[0] for l in path.read_text().splitlines() if l.startswith("nearest ")]
    assert len(key) == 1
    for w in (1, 2, 4, 8, 16):
        path.write_text(f"{key[0]} = {w}\n")
        mp.autotune_cache_load(str(path))
        assert torch.equal(mp.nearest(tree, q, c, filter=filt), want)
    mp.autotune_cache_clear()
