"""GPU: the last phase of a ROADMAP round (adjacency lists, degrees, start-goal
connectivity) against a sequential restatement on the host.  The two forms of
the planner share that phase, so comparing them does not check it.  A program of
its own includes the planner's source for its kernel and is linked with the
library's other objects."""
import glob
import os
import subprocess

import pytest

from paper_2609_30644_gb300 import build as B

pytestmark = pytest.mark.gpu

PROGRAM = r"""
#include "planner.cu"
#include <cstdio>
#include <random>

using namespace mrpop;

// Rounds of m new vertices over rcap rows; a new vertex lists up to per lower
// vertices, the share `ok` of them valid.  near: lists stay within the last
// `near` vertices (0: anywhere), so that the goal is reached late or never.
static bool rounds(int n_rounds, int m, int per, double ok, int near, int start, unsigned seed) {
    const int total = start + n_rounds * m, emax = (m + 2) * kKmax;
    std::mt19937 rng(seed);
    std::vector<int> adj((size_t)total * kKmax, -7), deg(total, 0);
    RmJob J{};
    J.rcap = total;
    RmJob *dJ = nullptr;
    bool good = !cudaMalloc(&J.adj, sizeof(int) * adj.size()) &&
                !cudaMalloc(&J.deg, sizeof(int) * total) && !cudaMalloc(&J.count, sizeof(int)) &&
                !cudaMalloc(&J.evalid, emax) && !cudaMalloc(&J.ea, sizeof(int) * emax) &&
                !cudaMalloc(&J.eb, sizeof(int) * emax) &&
                !cudaMalloc(&J.level, sizeof(int) * total) && !cudaMalloc(&J.conn, sizeof(int)) &&
                !cudaMalloc(&dJ, sizeof(RmJob));
    if (!good) return false;
    cudaMemcpy(J.adj, adj.data(), sizeof(int) * adj.size(), cudaMemcpyHostToDevice);
    cudaMemset(J.deg, 0, sizeof(int) * total);
    cudaMemset(J.conn, 0, sizeof(int));
    int n_old = start;
    auto push = [&](int x, int y) {
        if (deg[x] < kKmax) adj[(size_t)x * kKmax + deg[x]++] = y;
    };
    for (int r = 0; r < n_rounds && good; ++r) {
        const int n = n_old + m, first = n_old == 2 ? 0 : n_old, gathered = n - first;
        std::vector<int> ea(emax, -1), eb(emax, -1);
        std::vector<uint8_t> valid(emax, 0);
        for (int j = 0; j < gathered; ++j) {
            const int x = first + j, lo = near ? std::max(0, x - near) : 0;
            std::vector<int> list;
            for (int k = 0; k < per && x > lo; ++k) list.push_back(lo + (int)(rng() % (x - lo)));
            std::sort(list.begin(), list.end());
            list.erase(std::unique(list.begin(), list.end()), list.end());
            for (size_t k = 0; k < list.size() && k < (size_t)kKmax; ++k) {
                const int e = j * kKmax + (int)k;
                ea[e] = x;
                eb[e] = list[k];
                valid[e] = rng() % 1000 < ok * 1000;
            }
        }
        for (int e = 0; e < gathered * kKmax; ++e)
            if (valid[e] && ea[e] >= 0) push(ea[e], eb[e]), push(eb[e], ea[e]);
        std::vector<char> seen(n, 0);
        std::vector<int> queue{0};
        seen[0] = 1;
        for (size_t i = 0; i < queue.size(); ++i)
            for (int k = 0; k < deg[queue[i]]; ++k) {
                const int y = adj[(size_t)queue[i] * kKmax + k];
                if (!seen[y]) seen[y] = 1, queue.push_back(y);
            }
        J.m = gathered;
        J.first = first;
        J.n_old = n_old;
        cudaMemcpy(J.count, &n, sizeof(int), cudaMemcpyHostToDevice);
        cudaMemcpy(J.evalid, valid.data(), emax, cudaMemcpyHostToDevice);
        cudaMemcpy(J.ea, ea.data(), sizeof(int) * emax, cudaMemcpyHostToDevice);
        cudaMemcpy(J.eb, eb.data(), sizeof(int) * emax, cudaMemcpyHostToDevice);
        cudaMemcpy(dJ, &J, sizeof(RmJob), cudaMemcpyHostToDevice);
        k_rmb_link<<<dim3(1, 1), 256>>>(dJ);
        std::vector<int> gadj(adj.size()), gdeg(total);
        int conn = -1;
        good = !cudaDeviceSynchronize();
        cudaMemcpy(gadj.data(), J.adj, sizeof(int) * adj.size(), cudaMemcpyDeviceToHost);
        cudaMemcpy(gdeg.data(), J.deg, sizeof(int) * total, cudaMemcpyDeviceToHost);
        cudaMemcpy(&conn, J.conn, sizeof(int), cudaMemcpyDeviceToHost);
        good = good && gadj == adj && gdeg == deg && conn == (int)seen[1];
        if (!good)
            std::printf("round %d of %d new (%d listed, %g valid, near %d, start %d): adj %d deg %d "
                        "conn %d/%d\n", r, m, per, ok, near, start, gadj == adj, gdeg == deg, conn,
                        (int)seen[1]);
        n_old = n;
    }
    cudaFree(J.adj), cudaFree(J.deg), cudaFree(J.count), cudaFree(J.evalid), cudaFree(J.ea);
    cudaFree(J.eb), cudaFree(J.level), cudaFree(J.conn), cudaFree(dJ);
    return good;
}

int main() {
    bool ok = true;
    // gathered vertices at the edges of the 64-vertex tile; sparse lists, and
    // lists that fill every slot
    for (int m : {1, 2, 61, 62, 63, 64, 65, 126, 127, 128, 129, 200})
        for (int per : {1, 3, 40, 200}) ok = rounds(4, m, per, 0.6, 0, 2, 100 * m + per) && ok;
    ok = rounds(6, 64, 64, 0.0, 0, 2, 1) && ok;      // no valid edge: never connected
    ok = rounds(5, 300, 2, 0.9, 2, 2, 2) && ok;      // long chains: many search levels
    ok = rounds(3, 500, 2, 1.0, 1, 2, 3) && ok;      // one chain
    // up to the shared tables' 16,384 vertices, and above them
    ok = rounds(3, 128, 30, 0.7, 0, 16000, 4) && ok;
    ok = rounds(2, 64, 200, 0.7, 300, 16256, 5) && ok;
    ok = rounds(3, 64, 30, 0.7, 0, 16300, 6) && ok;
    return ok ? 0 : 1;
}
"""


def test_link_against_sequential(tmp_path):
    src, exe = tmp_path / "link.cu", tmp_path / "link"
    src.write_text(PROGRAM)
    objs = [o for o in sorted(glob.glob(os.path.join(B.BUILD, "*.o"))) if "planner" not in o]
    assert objs, "the library's objects are not built"
    subprocess.run([B.nvcc(), *B.NVCC_FLAGS, "-o", str(exe), str(src), *objs], check=True,
                   timeout=400)
    r = subprocess.run([str(exe)], capture_output=True, text=True, timeout=120)
    assert r.returncode == 0, r.stdout + r.stderr
