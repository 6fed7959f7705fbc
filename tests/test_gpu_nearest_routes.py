"""GPU: the routes of NEAREST give the same indices.  The small-batch scan is
checked against the oracle elsewhere; here the other routes are compared with
it, index for index."""
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


def _dev(a):
    return torch.from_numpy(np.ascontiguousarray(a)).cuda()


def _scan(mp, tree, q, c, n):
    """The scan, through batches that are too small for any other route."""
    return torch.cat([mp.nearest(tree, q[:, i:i + 32].contiguous(), c[i:i + 32].contiguous(),
                                 n_vertices=n) for i in range(0, q.shape[1], 32)])


def _inputs(D, n, Q, seed):
    lo, hi = -2.9 * np.ones(D), 2.9 * np.ones(D)
    tree = synth.random_tree_fast(D, n + 5, lo, hi, seed=seed)
    diag = float(np.sqrt(D) * 5.8)
    qs, cs = synth.nn_queries(D, Q, lo, hi, seed=seed + 1, budget_lo=0.3 * diag,
                              budget_hi=1.9 * diag)
    # exact ties: duplicated vertices, some with equal g, and queries on them
    k = min(n // 4, 40)
    tree[:, n - k:n] = tree[:, :k]
    tree[D, n - k:n - k // 2] += np.float32(0.5)
    kq = min(k, Q)
    qs[:, :kq] = tree[:D, :kq]
    return tree, qs, cs


# every padded instance, just above and at its rows, with a ragged last query
# block and slice
@pytest.mark.parametrize("D", [1, 2, 4, 5, 8, 12, 13, 15, 16, 17, 21, 22, 24, 25, 29, 32, 33, 35,
                               36, 37, 42, 44, 45, 49, 52, 53, 56, 57, 63, 64])
def test_large_batches_in_every_dimension(mp, D):
    n, Q = 3001, 4100
    tree, qs, cs = _inputs(D, n, Q, D)
    t, q, c = _dev(tree), _dev(qs), _dev(cs)
    want = _scan(mp, t, q, c, n)
    for filt in (0, 1):
        torch.testing.assert_close(mp.nearest(t, q, c, n_vertices=n, filter=filt), want,
                                   rtol=0, atol=0)


@pytest.mark.parametrize("D", [14, 35])
@pytest.mark.parametrize("what", ["inf_g", "neg_inf_g", "all_neg_inf_g", "inf_budget",
                                  "nan", "huge", "lowest", "equal_g", "offset", "tiny",
                                  "colossal", "scaled_down", "scaled_up"])
def test_large_batches_of_extreme_values(mp, D, what):
    n, Q = 2600, 4096
    tree, qs, cs = _inputs(D, n, Q, 7)
    if what == "inf_g":
        tree[D, ::3] = np.inf
    elif what == "neg_inf_g":
        tree[D, 5::11] = -np.inf
        cs[:7] = -np.float32(3e38)
    elif what == "all_neg_inf_g":
        tree[D] = -np.inf
    elif what == "inf_budget":
        cs[::2], cs[1::4] = np.inf, -np.inf
    elif what == "nan":
        tree[0, 3::7], tree[D, 4::9], qs[D - 1, ::13], cs[::5] = (np.nan,) * 4
    elif what == "huge":
        tree[1, ::17] = 3e38
        qs[1, 100] = np.float32(3e38)
        cs[100] = np.inf
    elif what == "lowest":
        cs[::2] = np.finfo(np.float32).min
    elif what == "equal_g":
        tree[D] = np.float32(1.5)
    elif what == "offset":              # large norms, small distances
        tree[:D] += np.float32(1000.0)
        qs += np.float32(1000.0)
    elif what == "tiny":                # below the filter's range: every pair decided exactly
        qs[3, 5] = np.float32(1e-25)
    elif what == "colossal":            # -2 q overflows
        qs[2, 9] = tree[2, 9] = np.float32(3e38)
        cs[9] = tree[D, 9] + np.float32(1.0)
    elif what in ("scaled_down", "scaled_up"):
        for a in (tree, qs, cs):
            a *= np.float32(1e-12 if what == "scaled_down" else 1e15)
    t, q, c = _dev(tree), _dev(qs), _dev(cs)
    torch.testing.assert_close(mp.nearest(t, q, c, n_vertices=n), _scan(mp, t, q, c, n),
                               rtol=0, atol=0)


# the scan's routes: one slice, a cluster of slices, slices with a second
# kernel; rows of 6, 7 and 8 with and without padding; ragged query tiles,
# steps and rows that are not 16-byte aligned
@pytest.mark.parametrize("D,n,Q", [(6, 1, 1), (7, 255, 64), (8, 257, 65), (9, 1023, 63), (14, 2048, 2),
                                   (13, 2049, 130), (28, 5003, 257), (35, 20001, 40), (64, 3001, 70),
                                   (3, 999, 2500), (1, 4000, 300)])
def test_scan_against_oracle(mp, orc, D, n, Q):
    tree, qs, cs = _inputs(D, n, Q, D + n) if n > 4 else (
        np.zeros((D + 1, 6), np.float32), np.ones((D, Q), np.float32), np.full(Q, 9.0, np.float32))
    t, q, c = _dev(tree), _dev(qs), _dev(cs)
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


# one block, clusters of 2 to 8 with ragged ranges, queries that fill a block's
# warps partly, lists that overflow k_max, and the two-kernel path (long lists,
# high dimensions)
@pytest.mark.parametrize("D,n,Q,k_max,delta", [
    (3, 1, 3, 4, 9.0), (7, 255, 9, 64, 2.5), (7, 257, 8, 16, 2.5), (7, 4097, 100, 32, 2.5),
    (4, 2048, 33, 64, 3.0), (10, 3000, 17, 0, 4.0), (11, 1500, 40, 7, 5.0), (16, 5000, 25, 64, 6.0),
    (17, 3000, 20, 64, 6.0), (7, 3000, 20, 65, 3.0), (7, 5, 2, 64, 0.0)])
def test_neighbors_against_oracle(mp, orc, D, n, Q, k_max, delta):
    rng = np.random.default_rng(D * n)
    tree = np.zeros((D + 1, n + 3), np.float32)
    tree[:D] = rng.uniform(-2.9, 2.9, (D, n + 3))
    qs = rng.uniform(-2.9, 2.9, (D, Q)).astype(np.float32)
    k = min(Q, n)
    qs[:, :k] = tree[:D, :k]                  # distance exactly zero
    idx, cnt = mp.neighbors(_dev(tree), _dev(qs), delta, k_max, n_vertices=n)
    idx, cnt = idx.cpu().numpy(), cnt.cpu().numpy()
    sub = np.ascontiguousarray(tree[:, :n])
    for i in range(Q):
        ref, rc, gap = orc.neighbors(sub, qs[:, i], np.float32(delta), k_max)
        if gap <= 1e-5 * delta and delta > 0:
            assert abs(int(cnt[i]) - rc) <= 2
            continue
        assert cnt[i] == rc
        np.testing.assert_array_equal(idx[i, :min(rc, k_max)], ref[:k_max])
        assert (idx[i, min(rc, k_max):] == -1).all()


@pytest.mark.parametrize("M", [0, 1, 2, 1024, 1025, 1026, 4097, 131073, 131074])
@pytest.mark.parametrize("D", [1, 6, 7, 8])
def test_path_cost_sizes(mp, M, D):
    rng = np.random.default_rng(M + D)
    buf = torch.from_numpy(rng.uniform(-2.9, 2.9, M * D + 3).astype(np.float32)).cuda()
    for off in (0, 1, 2):                     # 16-, 4- and 8-byte aligned rows
        path = buf[off:off + M * D].view(M, D)
        got = mp.path_cost(path).item()
        ref = (path[1:].double() - path[:-1].double()).norm(dim=1).sum().item()
        # FP32 segment lengths: (D + 3) roundings of 2^-24 each at most
        assert abs(got - ref) <= (D + 3) * 2.0 ** -24 * ref
        assert mp.path_cost(path).item() == got


@pytest.mark.parametrize("M", [16384, 16385, 16386, 17000])
def test_path_cost_cluster_limit(mp, M):
    path = torch.from_numpy(np.random.default_rng(M).uniform(-2.9, 2.9, (M, 14)).astype(np.float32)).cuda()
    got = mp.path_cost(path).item()
    ref = (path[1:].double() - path[:-1].double()).norm(dim=1).sum().item()
    assert abs(got - ref) <= 17 * 2.0 ** -24 * ref
