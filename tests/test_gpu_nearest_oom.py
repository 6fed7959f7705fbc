"""GPU: NEAREST without device memory to spare.  A program of its own, linked
with the library's objects, puts a fake in the place of the library's scratch
allocation that fails on request; nothing fills the device."""
import glob
import os
import subprocess

import pytest

from paper_2609_30644_gb300 import build as B

pytestmark = pytest.mark.gpu

SCRATCH = "_ZN5mrpop13scratch_allocEPPvmP11CUstream_st"   # mrpop::scratch_alloc

PROGRAM = r"""
#include <cstdio>
#include <cstdlib>
#include <vector>
#include <cuda_runtime.h>
#include "mrpop.h"

static bool fail = false;
static int refused = 0;
extern "C" cudaError_t __real_SCRATCH(void **, size_t, cudaStream_t);
extern "C" cudaError_t __wrap_SCRATCH(void **p, size_t n, cudaStream_t st) {
    if (!fail) return __real_SCRATCH(p, n, st);
    ++refused;
    return cudaErrorMemoryAllocation;
}

static bool run(int dim, int N, int Q) {
    std::vector<float> h((size_t)(dim + 1) * N), q((size_t)dim * Q), c(Q);
    srand(dim + N);
    for (float &x : h) x = (float)rand() / RAND_MAX;
    for (float &x : q) x = (float)rand() / RAND_MAX;
    for (float &x : c) x = 2.f + (float)rand() / RAND_MAX;
    float *dt, *dq, *dc;
    int64_t *out;
    std::vector<int64_t> want(Q), got(Q);
    if (cudaMalloc(&dt, h.size() * 4) || cudaMalloc(&dq, q.size() * 4) ||
        cudaMalloc(&dc, c.size() * 4) || cudaMalloc(&out, (size_t)Q * 8))
        return false;
    cudaMemcpy(dt, h.data(), h.size() * 4, cudaMemcpyHostToDevice);
    cudaMemcpy(dq, q.data(), q.size() * 4, cudaMemcpyHostToDevice);
    cudaMemcpy(dc, c.data(), c.size() * 4, cudaMemcpyHostToDevice);
    bool ok = true;
    for (int pass = 0; pass < 2; ++pass) {
        fail = pass == 1;
        refused = 0;
        cudaMemset(out, 0xff, (size_t)Q * 8);
        const mrpop_status s = mrpop_nearest(dt, N, N, dim, dq, dc, Q, out, nullptr);
        if (s != MRPOP_OK) std::printf("dim %d N %d Q %d: %s\n", dim, N, Q, mrpop_last_error());
        ok = ok && s == MRPOP_OK && refused == pass;  // the ordered copies only
        if (cudaMemcpy(pass ? got.data() : want.data(), out, (size_t)Q * 8, cudaMemcpyDeviceToHost))
            return false;
    }
    fail = false;
    long found = 0;
    for (int64_t v : want) found += v >= 0;
    cudaFree(dt), cudaFree(dq), cudaFree(dc), cudaFree(out);
    return ok && found > Q / 2 && want == got;
}

int main() {
    // slices of the tree: 30 and 9 (with scratch), 4
    return run(14, 400000, 600) && run(14, 40000, 2100) && run(35, 20000, 4500) ? 0 : 1;
}
"""


def test_ordered_path_falls_back_without_scratch(tmp_path):
    src, exe = tmp_path / "oom.cu", tmp_path / "oom"
    src.write_text(PROGRAM.replace("SCRATCH", SCRATCH))
    objs = sorted(glob.glob(os.path.join(B.BUILD, "*.o")))
    assert objs, "the library's objects are not built"
    subprocess.run([B.nvcc(), "-std=c++17", "-I", B.INCLUDE, *B.GENCODE, "-Xlinker",
                    f"--wrap={SCRATCH}", "-o", str(exe), str(src), *objs], check=True, timeout=300)
    r = subprocess.run([str(exe)], capture_output=True, text=True, timeout=120)
    assert r.returncode == 0, r.stdout + r.stderr
