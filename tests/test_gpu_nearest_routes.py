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
    qs[:, :k] = tree[:D, :k]
    return tree, qs, cs


# every padded instance, just above and at its rows, with a ragged last query
# block and slice
@pytest.mark.parametrize("D", [1, 2, 4, 5, 8, 12, 13, 15, 16, 17, 21, 22, 24, 25, 29, 32, 33, 35,
                               36, 37, 42, 44, 45, 49, 52, 53, 56, 57, 63, 64])
def test_large_batches_in_every_dimension(mp, D):
    n, Q = 3001, 2100
    tree, qs, cs = _inputs(D, n, Q, D)
    t, q, c = _dev(tree), _dev(qs), _dev(cs)
    want = _scan(mp, t, q, c, n)
    for filt in (0, 1):
        torch.testing.assert_close(mp.nearest(t, q, c, n_vertices=n, filter=filt), want,
                                   rtol=0, atol=0)


@pytest.mark.parametrize("D", [14, 35])
@pytest.mark.parametrize("what", ["inf_g", "neg_inf_g", "all_neg_inf_g", "inf_budget",
                                  "nan", "huge", "lowest", "equal_g"])
def test_large_batches_of_extreme_values(mp, D, what):
    n, Q = 2500, 2048
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
    t, q, c = _dev(tree), _dev(qs), _dev(cs)
    torch.testing.assert_close(mp.nearest(t, q, c, n_vertices=n), _scan(mp, t, q, c, n),
                               rtol=0, atol=0)
