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


def _scan_against_oracle(mp, orc, D, n, Q):
    if n > 4:
        lo, hi = -2.9 * np.ones(D), 2.9 * np.ones(D)
        diag = float(np.sqrt(D) * 5.8)
        tree = synth.random_tree_fast(D, n + 5, lo, hi, seed=D + n)
        qs, cs = synth.nn_queries(D, Q, lo, hi, seed=D + n + 1, budget_lo=0.3 * diag,
                                  budget_hi=1.9 * diag)
        k = min(n // 4, 40)                   # exact ties, some with equal g
        tree[:, n - k:n] = tree[:, :k]
        tree[D, n - k:n - k // 2] += np.float32(0.5)
        qs[:, :min(k, Q)] = tree[:D, :min(k, Q)]
    else:
        tree = np.zeros((D + 1, 6), np.float32)
        qs, cs = np.ones((D, Q), np.float32), np.full(Q, 9.0, np.float32)
    t, q, c = (torch.from_numpy(np.ascontiguousarray(a)).cuda() for a in (tree, qs, cs))
    got = mp.nearest(t, q, c, n_vertices=n).cpu().numpy()
    noalloc = torch.full((Q,), -7, dtype=torch.int64, device="cuda")
    assert mp.lib.mrpop_nearest_noalloc(t.data_ptr(), n, tree.shape[1], D, q.data_ptr(),
                                        c.data_ptr(), Q, noalloc.data_ptr(),
                                        torch.cuda.current_stream().cuda_stream) == 0
    np.testing.assert_array_equal(noalloc.cpu().numpy(), got)
    for i in range(0, Q, max(1, Q // 60)):
        ref, bd, sd, gap = orc.nearest(tree, qs[:, i], cs[i], n_vertices=n)
        # a different vertex only where FP32 cannot tell the two apart
        assert got[i] == ref or (np.isfinite(sd) and sd - bd <= 1e-5 * max(bd, 1e-30)) or \
            gap <= 1e-5 * max(1.0, abs(float(cs[i]))), (i, got[i], ref)


# few pairs, in pieces of 8 queries above 16 dimensions: every padded dimension at
# and above its rows, one slice and several, ragged slices and query groups
@pytest.mark.parametrize("D", [1, 4, 5, 8, 13, 16, 17, 20, 21, 24, 25, 28, 29, 32, 33, 48, 49, 64])
@pytest.mark.parametrize("n,Q", [(1, 1), (255, 9), (1024, 64), (2049, 33), (5003, 257), (40001, 7)])
def test_scan_of_few_pairs(mp, orc, D, n, Q):
    _scan_against_oracle(mp, orc, D, n, Q)


# the register tiles: one slice, clusters of slices, slices with a second kernel;
# rows of 6, 7 and 8 with and without padding; last steps of one and of all but one
# vertex; both sides of the lines between the two forms
@pytest.mark.parametrize("D,n,Q", [(7, 1025, 64), (8, 1500, 65), (9, 2047, 63), (32, 2048, 2),
                                   (33, 1025, 900), (64, 2048, 977), (13, 2049, 1220), (6, 257, 5100),
                                   (28, 2100, 1216), (28, 2100, 1217), (28, 5003, 600), (35, 2100, 400),
                                   (35, 2100, 410), (64, 3001, 900), (3, 1000, 3500), (6, 300, 12001),
                                   (64, 999, 2432), (64, 999, 2433), (17, 511, 2432), (17, 513, 2433),
                                   (14, 100003, 9), (12, 4095, 70),
                                   # clusters that fill the chip, one more and their scratch
                                   (8, 4000, 2304), (8, 4000, 2305), (14, 3000, 2944), (14, 3000, 2945),
                                   (6, 2000, 4736), (6, 2000, 4737), (4, 2000, 9729)])
def test_scan_in_tiles(mp, orc, D, n, Q):
    _scan_against_oracle(mp, orc, D, n, Q)


# one query on either side of its line to the ranges, and two
@pytest.mark.parametrize("D,n,Q", [(7, 24576, 1), (7, 24577, 1), (16, 40001, 1), (4, 40001, 1),
                                   (7, 40001, 2)])
@pytest.mark.parametrize("k_max", [8, 64])
def test_neighbors_of_few_queries(mp, orc, D, n, Q, k_max):
    rng = np.random.default_rng(D * n)
    tree = np.zeros((D + 1, n), np.float32)   # the last row is g, which is not read
    tree[:D] = rng.uniform(-2.9, 2.9, (D, n))
    qs = rng.uniform(-1.0, 1.0, (D, Q)).astype(np.float32)
    delta = np.float32({4: 0.7, 7: 1.8, 16: 5.0}[D])
    idx, cnt = mp.neighbors(torch.from_numpy(tree).cuda(), torch.from_numpy(qs).cuda(),
                            float(delta), k_max, dim=D)
    idx, cnt = idx.cpu().numpy(), cnt.cpu().numpy()
    for i in range(Q):
        ref, rc, gap = orc.neighbors(tree, qs[:, i], delta, k_max)
        if gap <= 1e-5 * delta:               # FP32 cannot decide a vertex
            assert abs(int(cnt[i]) - rc) <= 2
            continue
        assert cnt[i] == rc and rc > 0
        np.testing.assert_array_equal(idx[i, :min(rc, k_max)], ref[:k_max])
        assert (idx[i, min(rc, k_max):] == -1).all()


# odd dimensions (4-byte loads) on both sides of 350,000 floats in a path
@pytest.mark.parametrize("D,M", [(35, 10001), (35, 10002), (63, 5556), (63, 5557), (35, 16385),
                                 (23, 15218), (23, 15219)])
def test_path_cost_of_odd_dimensions(mp, D, M):
    p = torch.from_numpy(np.random.default_rng(M).uniform(-2.9, 2.9, (M, D)).astype(np.float32)).cuda()
    got = mp.path_cost(p).item()
    ref = (p[1:].double() - p[:-1].double()).norm(dim=1).sum().item()
    # FP32 segment lengths: (D + 3) roundings of 2^-24 each at most
    assert abs(got - ref) <= (D + 3) * 2.0 ** -24 * ref
    assert mp.path_cost(p).item() == got
