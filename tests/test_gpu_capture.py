"""GPU: a call that takes scratch memory can be captured into a CUDA graph as the
first call of a process.  Each runs in a process of its own; the graph's result
is compared with the call's after it."""
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

PROGRAM = """
import sys
sys.path.insert(0, {root!r})
import torch
import paper_2609_30644_gb300 as mp
torch.manual_seed(1)
def box(d, n):
    return (torch.rand(d, n, device="cuda") * 2 - 1) * 2.9
def nearest(dim, n, q):
    tree = box(dim + 1, n)
    tree[dim] = torch.rand(n, device="cuda") * 40
    queries, budgets = box(dim, q), 10 + 30 * torch.rand(q, device="cuda")
    return lambda: (mp.nearest(tree, queries, budgets),)
def neighbors(dim, n, q):
    tree, queries = box(dim, n), box(dim, q)
    return lambda: mp.neighbors(tree, queries, 2.0, 32)
def path_cost(dim, n):
    path = torch.rand(n, dim, device="cuda")
    return lambda: (mp.path_cost(path),)
call = {call}
torch.cuda.synchronize()
graph = torch.cuda.CUDAGraph()
with torch.cuda.graph(graph):
    got = call()
graph.replay()
torch.cuda.synchronize()
got = [g.clone() for g in got]
want = call()
torch.cuda.synchronize()
assert all(torch.equal(a, b) for a, b in zip(got, want))
"""


@pytest.mark.parametrize("call", ["nearest(35, 20000, 10000)",    # ordered copies
                                  "nearest(28, 50000, 200)",      # slices with a second kernel
                                  "neighbors(20, 4000, 100)", "path_cost(14, 65537)"])
def test_first_call_in_a_capture(call):
    r = subprocess.run([sys.executable, "-c", PROGRAM.format(root=ROOT, call=call)],
                       capture_output=True, text=True, timeout=300)
    assert r.returncode == 0, r.stderr[-2000:]
