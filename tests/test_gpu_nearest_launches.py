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


def _inputs(D, n, Q):
    diag = float(np.sqrt(D) * 5.8)
    lo, hi = -2.9 * np.ones(D), 2.9 * np.ones(D)
    tree = synth.random_tree_fast(D, n, lo, hi, seed=D)
    qs, cs = synth.nn_queries(D, Q, lo, hi, seed=D + 1, budget_lo=0.3 * diag, budget_hi=1.9 * diag)
    k = n // 4                                # exact ties, half of them with equal g
    tree[:, n - k:] = tree[:, :k]
    tree[D, n - k:n - k // 2] += np.float32(0.5)
    qs[:, :40] = tree[:D, :40]
    return [torch.from_numpy(np.ascontiguousarray(a)).cuda() for a in (tree, qs, cs)]


# every padded instance of the ordered path, just above and at its rows, at
# sizes whose work is above the line to it (6e8 pair coordinates)
@pytest.mark.parametrize("D", [1, 2, 4, 5, 8, 12, 13, 15, 16, 17, 22, 24, 25, 29, 32, 33, 35, 36,
                               37, 44, 45, 49, 52, 53, 56, 57, 64])
def test_padded_dimensions_above_the_work_line(mp, D):
    n = 8001
    Q = max(2049, int(6.2e8 / (n * D)) | 1)
    tree, q, c = _inputs(D, n, Q)
    assert mp.nearest_work(tree, q, c) < n * Q
    got = mp.nearest(tree, q, c)
    pick = torch.cat([torch.arange(40), torch.arange(40, Q, max(1, Q // 500)), torch.arange(Q - 9, Q)]).cuda()
    q, c = q[:, pick], c[pick]
    want = torch.cat([mp.nearest(tree, q[:, i:i + 64].contiguous(), c[i:i + 64].contiguous())
                      for i in range(0, q.shape[1], 64)])
    assert torch.equal(got[pick], want)


# below the line the scan serves the dimensions without a tensor-core filter,
# whichever filter is asked for
@pytest.mark.parametrize("D,n,Q", [(4, 2560, 4096), (16, 3500, 4096), (20, 2560, 8192),
                                   (35, 4001, 4097)])
def test_small_work_takes_the_scan(mp, D, n, Q):
    tree, q, c = _inputs(D, n, Q)
    assert mp.nearest_work(tree, q, c) == n * Q
    want = torch.cat([mp.nearest(tree, q[:, i:i + 64].contiguous(), c[i:i + 64].contiguous())
                      for i in range(0, Q, 64)])
    for filt in (0, 1):
        assert torch.equal(mp.nearest(tree, q, c, filter=filt), want)
