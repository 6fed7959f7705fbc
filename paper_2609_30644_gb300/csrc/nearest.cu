// Cost-filtered nearest neighbour (Alg. 2 NEAREST), radius query (Alg. 2
// NEIGHBORS) and path cost (Sec. III-A) over SoA state-cost trees.
//
// NEAREST, small batches: an exact scan of every pair in register tiles
// (nearest_scan_kernel) or, for few pairs, in finer pieces
// (nearest_small_kernel); when the tree is split across blocks (few queries,
// large tree), partial bests go to stream-ordered scratch and a second kernel
// reduces them.  Large batches take the budget-ordered path further down, with
// an FP32 expansion filter (or, as an option, one on the tensor cores) whose
// survivors are decided exactly.
#include <algorithm>
#include <atomic>
#include <cfloat>
#include <cmath>
#include <cooperative_groups.h>
#include <cuda_fp16.h>
#include <mutex>

#include "mrpop_internal.cuh"

namespace mrpop {
namespace {

constexpr unsigned kFull = 0xffffffffu;

struct Best {
    float d2;
    float g;
    int idx;
};

// Lexicographic (d^2, g, index); idx < 0 marks "none" (d2 = +inf).
__device__ __forceinline__ bool better(const Best &a, const Best &b) {
    if (a.d2 != b.d2) return a.d2 < b.d2;
    if (a.g != b.g) return a.g < b.g;
    return (unsigned)a.idx < (unsigned)b.idx;
}

__device__ __forceinline__ Best shfl_best(const Best &b, int off) {
    Best o;
    o.d2 = __shfl_xor_sync(kFull, b.d2, off);
    o.g = __shfl_xor_sync(kFull, b.g, off);
    o.idx = __shfl_xor_sync(kFull, b.idx, off);
    return o;
}

// Smallest of three floats (a NaN input is ignored while another is not NaN).
__device__ __forceinline__ float fmin3(float a, float b, float c) {
    float r;
    asm("min.f32 %0, %1, %2, %3;" : "=f"(r) : "f"(a), "f"(b), "f"(c));
    return r;
}

typedef unsigned long long f32x2_t;  // two floats, the first in the low half

__device__ __forceinline__ f32x2_t fma_f32x2(f32x2_t a, f32x2_t b, f32x2_t c) {
    f32x2_t r;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
    return r;
}
__device__ __forceinline__ f32x2_t add_f32x2(f32x2_t a, f32x2_t b) {
    f32x2_t r;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}
// acc += t * t, elementwise
__device__ __forceinline__ void acc_sq_f32x2(f32x2_t &acc, f32x2_t t) {
    asm("fma.rn.f32x2 %0, %1, %1, %0;" : "+l"(acc) : "l"(t));
}
__device__ __forceinline__ float f32x2_lo(f32x2_t v) { return __uint_as_float((unsigned)v); }
__device__ __forceinline__ float f32x2_hi(f32x2_t v) {
    return __uint_as_float((unsigned)(v >> 32));
}

// Source of the padding columns' folded norms: +inf never passes the filter.
__device__ const float g_f32_pad_inf = __builtin_inff();

__device__ __forceinline__ void cp_async4(float *dst, const float *src, bool ok) {
    const unsigned d = (unsigned)__cvta_generic_to_shared(dst);
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;" ::"r"(d), "l"(src),
                 "r"(ok ? 4 : 0)
                 : "memory");
}
// 16 bytes, of which the first src_bytes come from global memory and the
// rest are zero (both addresses 16-byte aligned)
__device__ __forceinline__ void cp_async16(float *dst, const float *src, int src_bytes) {
    const unsigned d = (unsigned)__cvta_generic_to_shared(dst);
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(d), "l"(src), "r"(src_bytes)
                 : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cp_async_wait() { asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory"); }
__device__ __forceinline__ void cp_async_wait_all() { asm volatile("cp.async.wait_group 0;" ::: "memory"); }


// ---------------------------------------------------------------------------
// NEAREST by an exact scan of every (query, vertex) pair, for batches that are
// too small to repay ordering the tree, and for mrpop_nearest_noalloc.
//
// A block takes 64 queries and a slice of the tree, a warp 8 of the queries and
// all of the block's vertices, 256 at a step: 8 vertices per lane, so a lane
// holds an 8 x 8 register tile of squared distances and every lane of a warp
// has the same queries.  Bound by the FMA pipe at two operations per
// coordinate of a pair (a difference and a fused multiply-add, both packed
// two to an instruction, each element rounded like the scalar one): a step of
// one coordinate is 64 packed instructions on 6 shared loads, of which the 4
// of the queries ({-q, -q} pairs) are broadcasts.  Coordinates come in chunks
// of 6 to 8 rows by cp.async, two chunks ahead.  The common case at
// the end of a step, no distance within the warp's best, costs a three-input
// minimum chain and one compare per query; what passes is checked for
// admissibility and kept per lane in shared memory, and one redux.sync per
// passing query shares the new best distance with the warp, an atomic minimum
// with the other slices of the tree (bounds, all bits set at the start; null:
// not shared), which read it once per step.
// One vertex per thread against 8 queries in registers, with the scalar forms
// and a padded template per dimension, took 122 us for 256 queries over
// 100,003 vertices in 28-D and a reduction of one thread per query 18 us;
// this takes 78 us and 5 us (FMA pipe at half of its peak: 1.4 steps' worth of
// each slice's 5 goes to its first bounds and its records).
// ---------------------------------------------------------------------------
constexpr int kScanThreads = 256;
constexpr int kScanQ = 64;       // queries per block
constexpr int kScanV = 256;      // vertices per step
constexpr int kScanStages = 3;
constexpr int kScanCluster = 8;  // slices of one cluster at most

inline size_t scan_smem_bytes(int dim, int rows) {
    // {-q, -q} [whole chunks][64], chunks [3][rows][256], g [4][256], best d2 /
    // vertex [8][256]
    const int padded = (dim + rows - 1) / rows * rows;
    return sizeof(float) * ((size_t)padded * 2 * kScanQ + kScanStages * rows * kScanV +
                            4 * kScanV + 2 * 8 * kScanThreads);
}

template <int kScanRows>
__global__ void __launch_bounds__(kScanThreads, 2)
nearest_scan_kernel(const float *__restrict__ tree, int N, int64_t ld, int dim,
                    const float *__restrict__ queries, const float *__restrict__ budgets, int Q,
                    int chunk, int vec, int64_t *__restrict__ out_idx,
                    Best *__restrict__ partial, unsigned *__restrict__ bounds) {
    extern __shared__ __align__(16) float scan_sm[];
    const int chunks = (dim + kScanRows - 1) / kScanRows;
    float *nq = scan_sm;                                   // [chunks * rows][2 * 64]
    float *xt = nq + (size_t)chunks * kScanRows * 2 * kScanQ;  // [3][rows][256]
    float *gt = xt + kScanStages * kScanRows * kScanV;     // [4][256]: issued two steps ahead
    float(*sb_d2)[kScanThreads] = reinterpret_cast<float(*)[kScanThreads]>(gt + 4 * kScanV);
    int(*sb_v)[kScanThreads] = reinterpret_cast<int(*)[kScanThreads]>(sb_d2 + 8);
    __shared__ float cq[kScanQ];
    __shared__ Best res[kScanQ];  // cluster launches: this slice's results
    const bool in_cluster = gridDim.y > 1 && !partial;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int q0 = blockIdx.x * kScanQ, nqb = min(kScanQ, Q - q0);
    const int vs = blockIdx.y * chunk, ve = (int)min((int64_t)N, (int64_t)vs + chunk);
    const int steps = (ve - vs + kScanV - 1) / kScanV;
    const float *grow = tree + (size_t)dim * ld;

    // chunk c of step s: rows [R c, R c + R) of 256 vertices, rows past the
    // dimension and columns past the slice zero; with the first chunk of a step also its g, +inf past the
    // slice (never admissible)
    int is = 0, ic = 0, ib = 0;  // next chunk to issue
    auto issue = [&]() {
        if (is < steps) {
            const int v0 = vs + is * kScanV, nv = min(kScanV, ve - v0);
            float *dst = xt + ib * kScanRows * kScanV;
            const int r0 = ic * kScanRows, rn = min(kScanRows, dim - r0);
            if (vec) {  // 16-byte rows and slices
                for (int i = tid; i < kScanRows * (kScanV / 4); i += kScanThreads) {
                    const int r = i / (kScanV / 4), j = 4 * (i % (kScanV / 4));
                    const int left = r < rn ? nv - j : 0;
                    cp_async16(dst + r * kScanV + j,
                               left > 0 ? tree + (size_t)(r0 + r) * ld + v0 + j : tree,
                               left >= 4 ? 16 : left > 0 ? 4 * left : 0);
                }
            } else {
#pragma unroll
                for (int r = 0; r < kScanRows; ++r) {
                    const bool ok = r < rn && tid < nv;
                    cp_async4(dst + r * kScanV + tid,
                              ok ? tree + (size_t)(r0 + r) * ld + v0 + tid : tree, ok);
                }
            }
            if (ic == 0)
                cp_async4(gt + (is & 3) * kScanV + tid, tid < nv ? grow + v0 + tid : &g_f32_pad_inf,
                          true);
            ib = ib == kScanStages - 1 ? 0 : ib + 1;
            if (++ic == chunks) {
                ic = 0;
                ++is;
            }
        }
        cp_async_commit();
    };
    issue();
    issue();
    for (int i = tid; i < chunks * kScanRows * kScanQ; i += kScanThreads) {
        const int d = i / kScanQ, j = i % kScanQ;
        const float v = j < nqb && d < dim ? -__ldg(queries + (size_t)d * Q + q0 + j) : 0.f;
        *reinterpret_cast<float2 *>(&nq[(size_t)d * 2 * kScanQ + 2 * j]) = make_float2(v, v);
    }
    if (tid < kScanQ) cq[tid] = tid < nqb ? __ldg(budgets + q0 + tid) : 0.f;
    float lim[8];  // the warp's best admissible distance; padding queries take none
#pragma unroll
    for (int r = 0; r < 8; ++r) {
        lim[r] = warp * 8 + r < nqb ? FLT_MAX * 2.f : -1.f;
        sb_d2[r][tid] = FLT_MAX * 2.f;
        sb_v[r][tid] = -1;
    }
    // the other slices' best distances of this warp's queries, a step old
    const int bq = q0 + warp * 8 + (lane & 7);
    unsigned other = 0x7f800000u;
    int buf = 0;
    for (int s = 0; s < steps; ++s) {
        if (bounds && bq < Q) other = min(__ldcg(bounds + bq), 0x7f800000u);
        f32x2_t acc2[8][4];
#pragma unroll
        for (int r = 0; r < 8; ++r)
#pragma unroll
            for (int p = 0; p < 4; ++p) acc2[r][p] = 0ull;
        for (int c = 0; c < chunks; ++c) {
            cp_async_wait<1>();
            __syncthreads();  // the chunk is visible; every thread is done with the one before it
            issue();
            const float *xs = xt + buf * kScanRows * kScanV + 4 * lane;
            const float *qs = nq + (size_t)c * kScanRows * 2 * kScanQ + 16 * warp;
            buf = buf == kScanStages - 1 ? 0 : buf + 1;
            // (a loop around the rows that is not unrolled makes the compiler
            // move the 64 accumulators between its iterations)
#pragma unroll
            for (int d = 0; d < kScanRows; ++d) {
                const ulonglong2 x0 = *reinterpret_cast<const ulonglong2 *>(xs + d * kScanV);
                const ulonglong2 x1 = *reinterpret_cast<const ulonglong2 *>(xs + d * kScanV + 128);
                const f32x2_t x[4] = {x0.x, x0.y, x1.x, x1.y};
                const ulonglong2 *a = reinterpret_cast<const ulonglong2 *>(qs + d * 2 * kScanQ);
#pragma unroll
                for (int h = 0; h < 4; ++h) {
                    const ulonglong2 ah = a[h];
#pragma unroll
                    for (int p = 0; p < 4; ++p) {
                        acc_sq_f32x2(acc2[2 * h][p], add_f32x2(x[p], ah.x));
                        acc_sq_f32x2(acc2[2 * h + 1][p], add_f32x2(x[p], ah.y));
                    }
                }
            }
        }
        unsigned rows = 0;
#pragma unroll
        for (int r = 0; r < 8; ++r) {
            lim[r] = fminf(lim[r], __uint_as_float(__shfl_sync(kFull, other, r)));
            const float m =
                fmin3(fmin3(f32x2_lo(acc2[r][0]), f32x2_hi(acc2[r][0]), f32x2_lo(acc2[r][1])),
                      fmin3(f32x2_hi(acc2[r][1]), f32x2_lo(acc2[r][2]), f32x2_hi(acc2[r][2])),
                      fminf(f32x2_lo(acc2[r][3]), f32x2_hi(acc2[r][3])));
            rows |= m <= lim[r] ? 1u << r : 0u;
        }
        const unsigned any = __reduce_or_sync(kFull, rows);
        const int v0 = vs + s * kScanV, nv = min(kScanV, ve - v0);
        const float *gs = gt + (s & 3) * kScanV;
#pragma unroll
        for (int r = 0; r < 8; ++r) {
            if (!((any >> r) & 1u)) continue;
            float d2[8];
#pragma unroll
            for (int p = 0; p < 4; ++p) {
                d2[2 * p] = f32x2_lo(acc2[r][p]);
                d2[2 * p + 1] = f32x2_hi(acc2[r][p]);
            }
            if (nv < kScanV)  // columns past the slice are zeros, which may lie near a query
#pragma unroll
                for (int k = 0; k < 8; ++k)
                    if (4 * lane + (k < 4 ? k : 124 + k) >= nv) d2[k] = FLT_MAX * 2.f;
            const float c = cq[warp * 8 + r];
            float bd = sb_d2[r][tid], lr = lim[r];
            int bv = sb_v[r][tid];
            // each round takes every lane's nearest remaining vertex within
            // the warp's best, which the round then tightens: one or two
            // rounds, where all 8 columns of a lane pass against a fresh bound
            for (;;) {
                const float m = fmin3(fmin3(d2[0], d2[1], d2[2]), fmin3(d2[3], d2[4], d2[5]),
                                      fminf(d2[6], d2[7]));
                const bool pass = m <= lr && m < FLT_MAX * 2.f;
                if (!__any_sync(kFull, pass)) break;
                if (pass) {
                    int at = 8;
#pragma unroll
                    for (int k = 7; k >= 0; --k)
                        if (d2[k] == m) at = k;
#pragma unroll
                    for (int k = 0; k < 8; ++k)
                        if (k == at) d2[k] = FLT_MAX * 2.f;
                    const int col = 4 * lane + (at < 4 ? at : 124 + at);
                    // filter of Alg. 2: g_v + |q - q_v| < c (strict); key (d^2,
                    // g, index): a lane's vertices come in index order within
                    // equal distances, so an equal one only wins by its g
                    const float g = gs[col];
                    if (m <= bd && g + __fsqrt_rn(m) < c &&
                        (m < bd || bv < 0 || g < __ldg(grow + bv))) {
                        bd = m;
                        bv = v0 + col;
                    }
                }
                // (distances are >= 0: their bits order like unsigned integers)
                lr = __uint_as_float(__reduce_min_sync(
                    kFull, min(__float_as_uint(lr), __float_as_uint(bd))));
            }
            sb_d2[r][tid] = bd;
            sb_v[r][tid] = bv;
            if (bounds && lane == 0 && lr < lim[r])
                atomicMin(bounds + q0 + warp * 8 + r, __float_as_uint(lr));
            lim[r] = lr;
        }
    }
#pragma unroll
    for (int r = 0; r < 8; ++r) {
        const int q = warp * 8 + r;
        if (q >= nqb) break;
        const int v = sb_v[r][tid];
        Best b{FLT_MAX * 2.f, FLT_MAX * 2.f, -1};
        if (v >= 0) b = Best{sb_d2[r][tid], __ldg(grow + v), v};
#pragma unroll
        for (int off = 16; off > 0; off >>= 1) {
            const Best o = shfl_best(b, off);
            if (better(o, b)) b = o;
        }
        if (lane == 0) {
            if (in_cluster)
                res[q] = b;
            else if (partial)
                partial[(size_t)(q0 + q) * gridDim.y + blockIdx.y] = b;
            else
                out_idx[q0 + q] = b.idx;
        }
    }
    if (!in_cluster) return;
    // the cluster's blocks hold all slices of these queries: each block decides
    // a share of them from the others' shared memory
    namespace cg = cooperative_groups;
    cg::cluster_group cl = cg::this_cluster();
    cl.sync();
    const int ranks = (int)cl.num_blocks(), rank = (int)cl.block_rank();
    for (int q = rank + ranks * tid; q < nqb; q += ranks * kScanThreads) {
        Best b = res[q];
        for (int k = 1; k < ranks; ++k) {
            const Best o = cl.map_shared_rank(res, (rank + k) % ranks)[q];
            if (better(o, b)) b = o;
        }
        out_idx[q0 + q] = b.idx;
    }
    cl.sync();  // no block ends while its results are read
}

// The slices' partial bests of a query (slice s of query q at q q_step + s s_step),
// one warp per query.  Launched so that its prologue overlaps the scan's tail;
// the wait comes before the first read.
__global__ void __launch_bounds__(256)
nearest_reduce_kernel(const Best *__restrict__ partial, int splits, int Q, int q_step, int s_step,
                      int64_t *__restrict__ out_idx) {
    cudaGridDependencySynchronize();
    const int q = blockIdx.x * 8 + (threadIdx.x >> 5), lane = threadIdx.x & 31;
    if (q >= Q) return;
    Best b{FLT_MAX * 2.f, FLT_MAX * 2.f, -1};
    for (int s = lane; s < splits; s += 32) {
        const Best o = partial[(size_t)q * q_step + (size_t)s * s_step];
        if (better(o, b)) b = o;
    }
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) {
        const Best o = shfl_best(b, off);
        if (better(o, b)) b = o;
    }
    if (lane == 0) out_idx[q] = b.idx;
}

inline mrpop_status reduce_launch(const Best *partial, int splits, int Q, int q_step, int s_step,
                                  int64_t *out_idx, cudaStream_t st) {
    cudaLaunchAttribute at{};
    at.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at.val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3((Q + 7) / 8);
    cfg.blockDim = dim3(256);
    cfg.stream = st;
    cfg.attrs = &at;
    cfg.numAttrs = 1;
    MRPOP_CUDA_TRY(cudaLaunchKernelEx(&cfg, nearest_reduce_kernel, partial, splits, Q, q_step,
                                      s_step, out_idx));
    return MRPOP_OK;
}

// Slices of the tree for Q queries: two blocks on every SM, whole steps each.
inline void scan_slices(int N, int Q, int sms, int64_t max_records, int *chunk, int *splits) {
    const int groups = (Q + kScanQ - 1) / kScanQ;
    int s = std::max(1, std::min(2 * sms / groups, (N + kScanV - 1) / kScanV));
    s = (int)std::min<int64_t>({(int64_t)s, max_records / Q, (int64_t)65535});
    const int64_t steps = ((int64_t)N + kScanV - 1) / kScanV;
    *chunk = (int)std::min<int64_t>(std::max<int64_t>(1, (steps + s - 1) / s) * kScanV,
                                    (int64_t)1 << 30);
    *splits = std::max(1, (int)(((int64_t)N + *chunk - 1) / *chunk));
}

// The scan of one batch in splits slices.  Up to kScanCluster slices run as
// one cluster per query tile where the chip holds all clusters at once
// (scan_in_clusters), which combines its own results: one launch and no scratch
// (2,000 vertices, 500 queries: 5 us less of host time than a second launch and
// its scratch cost).  Others write partial, splits records per query, for a
// second kernel; bounds (or null) is a word per query.
template <int R>
mrpop_status scan_launch(const float *tree, int N, int64_t ld, int dim, const float *queries,
                         const float *budgets, int Q, int chunk, int splits, int64_t *out_idx,
                         Best *partial, unsigned *bounds, cudaStream_t st) {
    static std::atomic<unsigned long long> raised{0};  // devices whose limit is raised
    int dev = 0;
    MRPOP_CUDA_TRY(cudaGetDevice(&dev));
    const unsigned long long bit = dev < 64 ? 1ull << dev : 0ull;
    if (!(raised.load() & bit)) {
        MRPOP_CUDA_TRY(cudaFuncSetAttribute(nearest_scan_kernel<R>,
                                            cudaFuncAttributeMaxDynamicSharedMemorySize,
                                            (int)scan_smem_bytes(MRPOP_MAX_LINKS, R)));
        raised.fetch_or(bit);
    }
    if (bounds) MRPOP_CUDA_TRY(cudaMemsetAsync(bounds, 0xff, sizeof(unsigned) * (size_t)Q, st));
    const int vec = ld % 4 == 0 && (reinterpret_cast<uintptr_t>(tree) & 15) == 0;
    cudaLaunchAttribute at{};
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3((Q + kScanQ - 1) / kScanQ, splits);
    cfg.blockDim = dim3(kScanThreads);
    cfg.dynamicSmemBytes = scan_smem_bytes(dim, R);
    cfg.stream = st;
    if (splits > 1 && !partial) {
        at.id = cudaLaunchAttributeClusterDimension;
        at.val.clusterDim.x = 1;
        at.val.clusterDim.y = splits;
        at.val.clusterDim.z = 1;
        cfg.attrs = &at;
        cfg.numAttrs = 1;
    }
    MRPOP_CUDA_TRY(cudaLaunchKernelEx(&cfg, nearest_scan_kernel<R>, tree, N, ld, dim, queries,
                                      budgets, Q, chunk, vec, out_idx, partial, bounds));
    return partial ? reduce_launch(partial, splits, Q, splits, 1, out_idx, st) : MRPOP_OK;
}

// Rows per chunk: 6, 7 or 8, whichever pads the dimension least (none for the
// multiples of 6, 7 and 8 that planar and 7-joint arms make), the largest of
// equals.
inline mrpop_status scan_rows(const float *tree, int N, int64_t ld, int dim, const float *queries,
                              const float *budgets, int Q, int chunk, int splits,
                              int64_t *out_idx, Best *partial, unsigned *bounds,
                              cudaStream_t st) {
    auto pad = [&](int r) { return (dim + r - 1) / r * r; };
    if (pad(8) <= std::min(pad(7), pad(6)))
        return scan_launch<8>(tree, N, ld, dim, queries, budgets, Q, chunk, splits, out_idx,
                              partial, bounds, st);
    if (pad(7) <= pad(6))
        return scan_launch<7>(tree, N, ld, dim, queries, budgets, Q, chunk, splits, out_idx,
                              partial, bounds, st);
    return scan_launch<6>(tree, N, ld, dim, queries, budgets, Q, chunk, splits, out_idx, partial,
                          bounds, st);
}

// ---------------------------------------------------------------------------
// The same scan for few pairs in more than 16 dimensions (small_scan), in finer
// pieces: a block takes 8 queries (staged in shared memory) and a slice of at
// least 1,024 vertices, a thread one vertex at a time against all 8.  Bound by
// latency: a block of the register tiles above works through 64 queries x 256
// vertices at least, alone on its SM while most SMs have none, and its time grows
// with the dimension (64-D, 450 vertices, 1,200 queries: 24.9 us a call in tiles,
// 16.9 here, which is the host's; 28-D, 2,100 x 1,200: 29.0 and 22.0).
// ---------------------------------------------------------------------------
constexpr int kSmallThreads = 256;
constexpr int kSmallQ = 8;

template <int DP>
__global__ void __launch_bounds__(kSmallThreads)
nearest_small_kernel(const float *__restrict__ tree, int N, int64_t ld, int dim,
                     const float *__restrict__ queries, const float *__restrict__ budgets, int Q,
                     int chunk, int64_t *__restrict__ out_idx, Best *__restrict__ partial) {
    __shared__ __align__(16) float qs[kSmallQ][DP];
    __shared__ float cs[kSmallQ];
    __shared__ Best wbest[kSmallThreads / 32][kSmallQ];
    const int q0 = blockIdx.x * kSmallQ;
    const int nq = min(kSmallQ, Q - q0);
    for (int i = threadIdx.x; i < kSmallQ * DP; i += blockDim.x) {
        const int j = i / DP, d = i % DP;
        qs[j][d] = (j < nq && d < dim) ? queries[(size_t)d * Q + q0 + j] : 0.f;
    }
    if (threadIdx.x < kSmallQ)
        cs[threadIdx.x] = threadIdx.x < nq ? budgets[q0 + threadIdx.x] : -FLT_MAX;
    __syncthreads();

    Best best[kSmallQ];
#pragma unroll
    for (int j = 0; j < kSmallQ; ++j) best[j] = Best{FLT_MAX * 2.f, FLT_MAX * 2.f, -1};

    const int vs = blockIdx.y * chunk;
    const int ve = min(N, vs + chunk);
    for (int v = vs + threadIdx.x; v < ve; v += blockDim.x) {
        float x[DP];
#pragma unroll
        for (int d = 0; d < DP; ++d) x[d] = d < dim ? __ldg(tree + (size_t)d * ld + v) : 0.f;
        const float g = __ldg(tree + (size_t)dim * ld + v);
#pragma unroll
        for (int j = 0; j < kSmallQ; ++j) {
            const float4 *q4 = reinterpret_cast<const float4 *>(qs[j]);
            float d2 = 0.f;
#pragma unroll
            for (int d = 0; d < DP / 4; ++d) {
                const float4 qq = q4[d];
                const float a0 = qq.x - x[4 * d], a1 = qq.y - x[4 * d + 1];
                const float a2 = qq.z - x[4 * d + 2], a3 = qq.w - x[4 * d + 3];
                d2 = fmaf(a0, a0, d2);
                d2 = fmaf(a1, a1, d2);
                d2 = fmaf(a2, a2, d2);
                d2 = fmaf(a3, a3, d2);
            }
            if (d2 <= best[j].d2) {
                // filter of Alg. 2: g_v + |q - q_v| < c (strict)
                if (g + __fsqrt_rn(d2) < cs[j] && (d2 < best[j].d2 || g < best[j].g)) {
                    best[j].d2 = d2;
                    best[j].g = g;
                    best[j].idx = v;
                }
            }
        }
    }

    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
#pragma unroll
    for (int j = 0; j < kSmallQ; ++j) {
        Best b = best[j];
#pragma unroll
        for (int off = 16; off > 0; off >>= 1) {
            const Best o = shfl_best(b, off);
            if (better(o, b)) b = o;
        }
        if (lane == 0) wbest[warp][j] = b;
    }
    __syncthreads();
    if (threadIdx.x < nq) {
        const int j = threadIdx.x;
        Best b = wbest[0][j];
        for (int w = 1; w < kSmallThreads / 32; ++w)
            if (better(wbest[w][j], b)) b = wbest[w][j];
        if (partial)
            partial[(size_t)blockIdx.y * Q + q0 + j] = b;
        else
            out_idx[q0 + j] = b.idx;
    }
}

// Slices of the tree: 8 blocks on every SM, of 1,024 vertices at least.
inline void small_slices(int N, int Q, int sms, int64_t max_records, int *chunk, int *splits) {
    const int64_t n = N, groups = ((int64_t)Q + kSmallQ - 1) / kSmallQ, target = (int64_t)sms * 8;
    int64_t s = 1;
    if (groups < target && n > 4 * kSmallThreads)
        s = std::min((target + groups - 1) / groups, (n + 4 * kSmallThreads - 1) / (4 * kSmallThreads));
    s = std::max<int64_t>(1, std::min<int64_t>({s, max_records / Q, 65535}));
    const int64_t c = std::max<int64_t>(
        kSmallThreads, ((n + s - 1) / s + kSmallThreads - 1) / kSmallThreads * kSmallThreads);
    *chunk = (int)std::min<int64_t>(c, (int64_t)1 << 30);
    *splits = (int)std::max<int64_t>(1, (n + *chunk - 1) / *chunk);
}

template <int DP>
mrpop_status small_launch(const float *tree, int N, int64_t ld, int dim, const float *queries,
                          const float *budgets, int Q, int chunk, int splits, int64_t *out_idx,
                          Best *partial, cudaStream_t st) {
    nearest_small_kernel<DP><<<dim3((Q + kSmallQ - 1) / kSmallQ, splits), kSmallThreads, 0, st>>>(
        tree, N, ld, dim, queries, budgets, Q, chunk, out_idx, partial);
    MRPOP_CUDA_TRY(cudaGetLastError());
    return partial ? reduce_launch(partial, splits, Q, 1, Q, out_idx, st) : MRPOP_OK;
}

// By the dimension in whole float4s; partial (more than one slice) or null.
inline mrpop_status small_dims(const float *tree, int N, int64_t ld, int dim, const float *queries,
                               const float *budgets, int Q, int chunk, int splits,
                               int64_t *out_idx, Best *partial, cudaStream_t st) {
#define MRPOP_SMALL_DIM(D)                                                                    \
    if (dim <= D)                                                                             \
        return small_launch<D>(tree, N, ld, dim, queries, budgets, Q, chunk, splits, out_idx, \
                               partial, st)
    MRPOP_SMALL_DIM(20);
    MRPOP_SMALL_DIM(24);
    MRPOP_SMALL_DIM(28);
    MRPOP_SMALL_DIM(32);
    MRPOP_SMALL_DIM(48);
    MRPOP_SMALL_DIM(64);
#undef MRPOP_SMALL_DIM
    return set_error(MRPOP_EINVAL, "nearest: dimension %d", dim);
}

// Whether a scan of N vertices for Q queries takes the finer pieces: where their
// blocks are one wave (two per SM fit of more than 32 dimensions, three below).
// Tiles / pieces (us): up to 1,024 vertices, one launch of either, 64-D 450 x 2,400
// 24.9 / 17.7, 450 x 4,000 25.1 / 31.1, 28-D 1,024 x 2,400 22.8 / 18.2, x 4,000 23.1 /
// 31.1.  Up to 2,048 the tiles are one cluster launch and the pieces two kernels
// and their scratch (28-D, 1,500 x 700 18.2 / 23.0; 64-D 24.0 / 25.2).  Above, both
// are two kernels (28-D, 10,000 x 300 25.8 / 25.2, 3,000 x 1,200 29.1 / 25.2; 64-D,
// 10,000 x 64 27.6 / 23.4, but beyond a block per SM 5,000 x 300 26.7 / 29.4).  Up to
// 16 dimensions the tiles are bound by the host's call there.
inline bool small_scan(int dim, int N, int Q, int sms, int64_t max_records) {
    if (dim <= 16 || (N > 4 * kSmallThreads && N <= kScanCluster * kScanV)) return false;
    int chunk = 0, splits = 1;
    small_slices(N, Q, sms, max_records, &chunk, &splits);
    const int per_sm = N <= 4 * kSmallThreads ? 2 : dim <= 32 ? 3 : 1;
    return ((int64_t)Q + kSmallQ - 1) / kSmallQ * splits <= (int64_t)per_sm * sms;
}

// Whether the scan's slices run as clusters of one query tile each.  The blocks of
// a cluster share a GPC, so a chip of two blocks on each of 152 SMs holds 36
// clusters of 8 at once, 38 of 7, 46 of 6, 58 of 5, 74 of 4, 97 of 3; one more
// is a second wave (14-D, 12,188 vertices in 6 slices, 3,000 queries, 47 clusters:
// 91.1 us, with scratch 63.2; 8,092 in 4, 4,500 queries, 71 clusters: 64.1 and 64.4).
inline mrpop_status scan_in_clusters(int splits, int Q, bool *out) {
    static std::atomic<int> active[64][kScanCluster + 1];  // of the device; 0: not asked yet
    *out = splits <= kScanCluster;
    if (!*out || splits <= 1) return MRPOP_OK;
    int dev = 0;
    MRPOP_CUDA_TRY(cudaGetDevice(&dev));
    int n = dev < 64 ? active[dev][splits].load() : 0;
    if (n == 0) {
        // the largest tables, of which two blocks still fit an SM
        const size_t smem = scan_smem_bytes(MRPOP_MAX_LINKS, 8);
        MRPOP_CUDA_TRY(cudaFuncSetAttribute(nearest_scan_kernel<8>,
                                            cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
        cudaLaunchAttribute at{};
        at.id = cudaLaunchAttributeClusterDimension;
        at.val.clusterDim.x = 1;
        at.val.clusterDim.y = splits;
        at.val.clusterDim.z = 1;
        cudaLaunchConfig_t cfg{};
        cfg.gridDim = dim3(1, splits);
        cfg.blockDim = dim3(kScanThreads);
        cfg.dynamicSmemBytes = smem;
        cfg.attrs = &at;
        cfg.numAttrs = 1;
        MRPOP_CUDA_TRY(cudaOccupancyMaxActiveClusters(&n, nearest_scan_kernel<8>, &cfg));
        if (dev < 64) active[dev][splits].store(n);
    }
    *out = (Q + kScanQ - 1) / kScanQ <= n;
    return MRPOP_OK;
}

inline mrpop_status nearest_scan(const float *tree, int N, int64_t ld, int dim,
                                 const float *queries, const float *budgets, int Q,
                                 int64_t *out_idx, cudaStream_t st, bool no_scratch) {
    int dev = 0, sms = 1, chunk = 0, splits = 1;
    MRPOP_CUDA_TRY(cudaGetDevice(&dev));
    MRPOP_CUDA_TRY(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
    Best *partial = nullptr;
    if (!no_scratch && small_scan(dim, N, Q, sms, INT64_MAX)) {
        small_slices(N, Q, sms, INT64_MAX, &chunk, &splits);
        if (splits > 1)
            MRPOP_CUDA_TRY(scratch_alloc((void **)&partial, sizeof(Best) * (size_t)splits * Q, st));
        const mrpop_status s = small_dims(tree, N, ld, dim, queries, budgets, Q, chunk, splits,
                                          out_idx, partial, st);
        if (partial) cudaFreeAsync(partial, st);
        return s;
    }
    scan_slices(N, Q, sms, no_scratch ? (int64_t)kScanCluster * Q : INT64_MAX, &chunk, &splits);
    const size_t records = (size_t)splits * Q;
    bool clusters = true;
    if (!no_scratch) {
        const mrpop_status s = scan_in_clusters(splits, Q, &clusters);
        if (s != MRPOP_OK) return s;
    }
    if (!clusters)
        MRPOP_CUDA_TRY(scratch_alloc((void **)&partial,
                                     sizeof(Best) * records + sizeof(unsigned) * (size_t)Q, st));
    const mrpop_status s =
        scan_rows(tree, N, ld, dim, queries, budgets, Q, chunk, splits, out_idx, partial,
                  partial ? reinterpret_cast<unsigned *>(partial + records) : nullptr, st);
    if (partial) cudaFreeAsync(partial, st);
    return s;
}

// ---------------------------------------------------------------------------
// NEAREST filter on the tensor cores.  The expansion
//   e(q, x) = |q|^2 + |x|^2 - 2 q.x
// is one contraction over D + 2 terms once the norms ride along as two extra
// coordinates: A[q] = (-2 q, 1, |q|^2) and B[x] = (x, |x|^2 (1 - kTc), 1),
// zero-padded to K.  A warp owns 32 queries (two 16-row m-tiles, A fragments
// in registers for the whole kernel) and walks the block's shared-memory
// vertex tile 8 vertices at a time with ldmatrix and mma.sync; the
// accumulators are the filter values, compared in registers against the
// running bound of their query.  Two operand types:
//
//  - FP16 for D + 2 <= 16 (nearest_tc16_kernel: one m16n8k16 per m-tile and
//    8 vertices).  The coordinates are first multiplied by a power of two 2^s
//    (exact), chosen from the largest coordinate magnitude of the batch so
//    that every scaled coordinate is below 16 and every scaled squared norm
//    below 256 D: the operands stay inside FP16's range.  Rounding to FP16
//    costs at most 2^-11 of an operand, or the operand itself when it is
//    below 2^-14 (a flush); with scaled coordinates below 16 the flushes add
//    less than 48 D 2^-14 + 2^-13 < kAbs = 2^-4 in all.
//  - TF32 for larger D (nearest_tc_kernel: m16n8k8 steps).  TF32 keeps 10 of
//    the 23 stored mantissa bits (truncation or rounding: 2^-10 of an
//    operand); there is no scaling, and every nonzero coordinate must lie in
//    [2^-60, 2^60] (normal products, no overflow).
//
// Products are exact and the FP32 accumulation error stays below 2^-14 of
// sum |a_k b_k| for K <= 32.  With sum |a_k b_k| <= 2 (|q|^2 + |x|^2) the
// computed value is within 1.0625 * 2^-9 (FP16; 1.04 * 2^-8 for TF32) of
// (|q|^2 + |x|^2), plus kAbs for FP16, from e (scaled units).  The vertex half
// of that error is taken out of B (kTc), the query half goes into the bound
// (kTq |q|^2).  The exact FP32 squared distance (sum of fmaf((q_d - x_d)^2))
// is within 4 (D + 2) u d^2 of the true one (u = 2^-24), so a bound built from
// the exact distance d2 of any admissible vertex as
//   lim = (d2 2^2s (1 + 4 (D + 2) u) + kTq |q|^2 + kAbs) (1 + 4 u)
// is never below the computed filter value of the true nearest vertex.  Every
// vertex that passes is re-evaluated with the exact formula on the unscaled
// FP32 coordinates, which alone decides: the results equal the plain scan's.
// The ordering pass flags inputs outside the operand type's range (NaN and
// infinities always) and the kernel then sends every pair to the exact check.
constexpr int kTcWarps = 8;
constexpr int kSliceAlign = 256;           // tree slices are whole tensor-core tiles
constexpr int kTcThreads = kTcWarps * 32;
constexpr int kTcQueries = kTcWarps * 32;  // queries per block
constexpr float kTc = 1.125f / 256.f;      // TF32: folded into |x|^2
constexpr float kTq = 1.25f / 256.f;       // TF32: widening by |q|^2
constexpr float kTc16 = 1.125f / 512.f;    // FP16: folded into |x|^2
constexpr float kTq16 = 1.25f / 512.f;     // FP16: widening by |q|^2
constexpr float kAbs16 = 1.f / 16.f;       // FP16: flushed operands (scaled units)

template <int DIM>
struct TcShape {
    static constexpr int K = ((DIM + 2 + 7) / 8) * 8;  // contraction length
    static constexpr int KS = K / 8;                   // m16n8k8 steps
    static constexpr int CH = K / 4;                   // 16-byte chunks per vertex row
    static constexpr int VT = K <= 16 ? 256 : 128;     // vertices per tile (16 KB)
};

// Chunk swizzle of a vertex row: the 8 rows one ldmatrix reads (8 consecutive
// vertices, one chunk each) land in 8 distinct 16-byte bank groups.
template <int CH>
__device__ __forceinline__ int tc_swz(int v) {
    if (CH == 8) return v & 7;
    if (CH == 4) return (v >> 1) & 3;
    return (v >> 2) & 1;  // CH = 2 or 6
}

__device__ __forceinline__ void mma_tf32(float (&d)[4], const unsigned (&a)[4], unsigned b0,
                                         unsigned b1) {
    asm("mma.sync.aligned.m16n8k8.row.col.f32.tf32.tf32.f32 {%0, %1, %2, %3}, "
        "{%4, %5, %6, %7}, {%8, %9}, {%0, %1, %2, %3};"
        : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
        : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}

__device__ __forceinline__ void ldsm_x4(unsigned addr, unsigned &r0, unsigned &r1, unsigned &r2,
                                        unsigned &r3) {
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0, %1, %2, %3}, [%4];"
                 : "=r"(r0), "=r"(r1), "=r"(r2), "=r"(r3)
                 : "r"(addr)
                 : "memory");
}
__device__ __forceinline__ void ldsm_x2(unsigned addr, unsigned &r0, unsigned &r1) {
    asm volatile("ldmatrix.sync.aligned.m8n8.x2.shared.b16 {%0, %1}, [%2];"
                 : "=r"(r0), "=r"(r1)
                 : "r"(addr)
                 : "memory");
}

// Pieces shared by both filter kernels.
//
// Stage the block's kTcQueries queries (SoA rows of the ordered batch) in
// shared memory, one per thread (kTcThreads == kTcQueries).
template <int DIM>
__device__ __forceinline__ void tc_stage_queries(float (*qsm)[kTcQueries],
                                                 const float *__restrict__ queries, int Q, int qb) {
    const int j = threadIdx.x;
    const bool ok = qb + j < Q;
#pragma unroll
    for (int d = 0; d < DIM; ++d) qsm[d][j] = ok ? __ldg(queries + (size_t)d * Q + qb + j) : 0.f;
}

// Smallest g of the tree slice [vs, ve) (row DIM of the ordered tree), for
// every thread of the block: an admissible vertex of the slice has
// |q - x| < c - that minimum.
template <int DIM>
__device__ __forceinline__ float tc_slice_gmin(const float *__restrict__ tree, int ldt, int vs,
                                               int ve, float *red_g) {
    float gm = FLT_MAX;
#pragma unroll 4
    for (int v = vs + threadIdx.x; v < ve; v += kTcThreads)
        gm = fminf(gm, __ldg(tree + (size_t)DIM * ldt + v));
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) gm = fminf(gm, __shfl_xor_sync(kFull, gm, o));
    if ((threadIdx.x & 31) == 0) red_g[threadIdx.x >> 5] = gm;
    __syncthreads();
#pragma unroll
    for (int k = 0; k < kTcWarps; ++k) gm = fminf(gm, red_g[k]);
    return gm;
}

// The four lanes of a quad hold the same four rows (queries row_q(r)), each
// with the best of its own vertex columns, as a position in the g order:
// translate to original indices (perm), combine by key, and let lane
// tig == 0 write the slice's partial bests.
// Where a budget-ordered filter block finishes its query block: the slice
// blocks of query block b count themselves in qdone[b]; the last one to
// finish reduces the partial bests of every slice, best key first, and writes
// the original query's index.
struct NnFinish {
    int *qdone;            // [query blocks] slices finished (zero before the filter)
    const int *qperm;      // ordered query -> original query index
    int64_t *out_idx;      // [Q] by original query index
};

// No slice of the block has work (its cut is empty): no query of it has an
// admissible vertex.
__device__ __forceinline__ void nn_write_none(const NnFinish &fin, int qb, int Q) {
    for (int j = threadIdx.x; j < kTcQueries; j += blockDim.x)
        if (qb + j < Q) fin.out_idx[fin.qperm[qb + j]] = -1;
}

// Called by every thread of a slice block after its partial bests are
// written; ns = slice blocks of this query block that have work.
__device__ __forceinline__ void nn_finish(const Best *partial, const NnFinish &fin, int qblk,
                                          int ns, int qb, int Q) {
    __shared__ int s_last;
    __threadfence();  // this thread's partial records, before the count
    __syncthreads();
    if (threadIdx.x == 0) s_last = atomicAdd(fin.qdone + qblk, 1) == ns - 1;
    __syncthreads();
    if (!s_last) return;
    __threadfence();
    for (int j = threadIdx.x; j < kTcQueries; j += blockDim.x) {
        const int q = qb + j;
        if (q >= Q) continue;
        Best b{FLT_MAX * 2.f, FLT_MAX * 2.f, -1};
        for (int y = 0; y < ns; ++y) {
            const Best *rec = partial + (size_t)y * Q + q;
            const Best o{__ldcg(&rec->d2), __ldcg(&rec->g), __ldcg(&rec->idx)};
            if (better(o, b)) b = o;
        }
        fin.out_idx[fin.qperm[q]] = b.idx;
    }
}

template <typename RowQ>
__device__ __forceinline__ void tc_write_rows(Best (&best)[4], const int *__restrict__ perm,
                                              RowQ row_q, int Q, Best *__restrict__ partial) {
#pragma unroll
    for (int r = 0; r < 4; ++r) {
        if (best[r].idx >= 0) best[r].idx = __ldg(perm + best[r].idx);
#pragma unroll
        for (int o = 1; o <= 2; o <<= 1) {
            const Best other = shfl_best(best[r], o);
            if (better(other, best[r])) best[r] = other;
        }
        const int q = row_q(r);
        if ((threadIdx.x & 3) == 0 && q < Q) partial[(size_t)blockIdx.y * Q + q] = best[r];
    }
}

// Inputs: the g-ordered tree (SoA rows of stride ldt) with perm (ordered ->
// original index), the budget-ordered queries, cut (vertices each query block
// scans), the shared bound seed (see below); *exhaustive != 0 turns the filter
// off.  Block (x, y) takes query block b = gridDim.x - 1 - x (queries
// [256 b, 256 b + 256)) and the tree slice [y chunk, (y + 1) chunk) cut at
// cut[b]; its partial bests go to partial[y][q], and the query block's last
// slice block to finish reduces them (nn_finish).
template <int DIM>
__global__ void __launch_bounds__(kTcThreads)
nearest_tc_kernel(const float *__restrict__ tree, int N, int ldt, const float *__restrict__ queries,
                  const float *__restrict__ budgets, int Q, int chunk,
                  Best *__restrict__ partial, const int *__restrict__ perm,
                  const int *__restrict__ cut, float *__restrict__ seed,
                  const int *__restrict__ exhaustive, NnFinish fin) {
    using S = TcShape<DIM>;
    constexpr int K = S::K, KS = S::KS, CH = S::CH, VT = S::VT;
    __shared__ __align__(16) float xt[VT * K];  // vertex rows, swizzled chunks
    __shared__ float gt[VT];
    __shared__ float qsm[DIM][kTcQueries];      // the block's queries (exact checks)
    __shared__ float red_g[kTcWarps];
    constexpr float kU = 5.9604645e-8f;            // 2^-24
    constexpr float kC1 = 4.f * (DIM + 2.f) * kU;  // exact-distance relative error
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int grp = lane >> 2, tig = lane & 3;
    // query blocks in descending budget order: the blocks with the longest
    // tree prefixes start first and the short ones fill the last wave
    const int qblk = gridDim.x - 1 - blockIdx.x;
    const int qb = qblk * kTcQueries;
    const int cut_q = min(N, cut[qblk]);
    const int vs = blockIdx.y * chunk;
    const int ve = min(cut_q, vs + chunk);
    if (vs >= ve) {  // no partial record: this slice is not counted
        if (blockIdx.y == 0) nn_write_none(fin, qb, Q);
        return;
    }
    const bool exact_only = *exhaustive != 0;

    tc_stage_queries<DIM>(qsm, queries, Q, qb);
    __syncthreads();
    // rows of this thread: slot r = 2 * mt + h is query qb + 32 warp + 16 mt + grp + 8 h
    auto row_l = [&](int r) { return warp * 32 + (r >> 1) * 16 + grp + (r & 1) * 8; };
    auto row_q = [&](int r) { return qb + row_l(r); };
    float cq[4], qn[4], lim[4];
    Best best[4];
    unsigned a[2][KS][4];
#pragma unroll
    for (int r = 0; r < 4; ++r) {
        const int q = row_q(r);
        const bool ok = q < Q;
        float n2 = 0.f;
#pragma unroll
        for (int d = 0; d < DIM; ++d) {
            const float v = qsm[d][row_l(r)];
            n2 = fmaf(v, v, n2);
        }
        qn[r] = n2;
        cq[r] = ok ? budgets[q] : -FLT_MAX;  // nothing is admissible for padding
        best[r] = Best{FLT_MAX * 2.f, FLT_MAX * 2.f, -1};
        lim[r] = FLT_MAX * 2.f;
    }
    // A fragments: a0 (row grp, k tig), a1 (row grp + 8, k tig), a2/a3 the same rows at k + 4
#pragma unroll
    for (int mt = 0; mt < 2; ++mt) {
#pragma unroll
        for (int ks = 0; ks < KS; ++ks) {
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                const int r = 2 * mt + (i & 1);
                const int q = row_q(r);
                const int k = 8 * ks + tig + 4 * (i >> 1);
                float v = 0.f;
                if (k < DIM)
                    v = q < Q ? -2.f * qsm[k][row_l(r)] : 0.f;
                else if (k == DIM)
                    v = 1.f;
                else if (k == DIM + 1)
                    v = qn[r];
                a[mt][ks][i] = __float_as_uint(v);
            }
        }
    }
    unsigned *const shared_lim = reinterpret_cast<unsigned *>(seed);
    auto widen = [&](int r, float sd) {
        if (sd <= FLT_MAX) lim[r] = fminf(lim[r], fmaf(sd, 1.f + kC1, kTq * qn[r]) * (1.f + 4.f * kU));
    };
    unsigned pend[4];
#pragma unroll
    for (int r = 0; r < 4; ++r) {
        const int q = row_q(r);
        pend[r] = q < Q ? __ldcg(shared_lim + q) : 0x7f800000u;
        widen(r, __uint_as_float(pend[r]));
    }
    {
        // an admissible vertex of this slice has |q - x| < c - g_min(slice)
        const float gm = tc_slice_gmin<DIM>(tree, ldt, vs, ve, red_g);
#pragma unroll
        for (int r = 0; r < 4; ++r) {
            if (!(cq[r] > gm)) {
                lim[r] = -FLT_MAX * 2.f;
            } else if (exact_only) {
                lim[r] = FLT_MAX * 2.f;
            } else {
                const float t = __fsub_ru(cq[r], gm);
                const float b2 = __fmul_ru(t, t);
                lim[r] = fminf(lim[r], fmaf(b2, 1.f + kC1, kTq * qn[r]) * (1.f + 4.f * kU));
            }
        }
    }
    const unsigned xt_s = (unsigned)__cvta_generic_to_shared(xt);
    // ldmatrix row addresses of this lane: matrix (lane >> 3) of a pair of
    // k-steps, vertex row (lane & 7) of the 8-vertex n-tile
    const int lrow = lane & 7, lmat = lane >> 3;
    // The next tile's vertex (coordinates and g) is loaded into registers
    // while the current tile is being scanned, so that the load latency
    // overlaps the tensor-core work; 32-bit element indices keep the per-row
    // offsets cheap (N (D + 1) < 2^31).
    const int t_ld = threadIdx.x & (VT - 1);  // VT < kTcThreads: two threads per row store the same values
    float px[DIM + 1];
    auto prefetch = [&](int v0n) {
        const bool ok = t_ld < min(VT, ve - v0n);
        const unsigned base = (unsigned)(v0n + t_ld);
#pragma unroll
        for (int d = 0; d <= DIM; ++d) px[d] = ok ? __ldg(tree + (base + (unsigned)d * (unsigned)ldt)) : 0.f;
        if (!ok) px[DIM] = FLT_MAX * 2.f;  // padding vertex: g = +inf
    };
    prefetch(vs);
    for (int v0 = vs; v0 < ve; v0 += VT) {
        const int nv = min(VT, ve - v0);
        __syncthreads();
        {
            // one vertex row per thread: coordinates, folded norm, 1, zero pad
            float *row = xt + t_ld * K;
            const int sw = tc_swz<CH>(t_ld);
            const bool ok = t_ld < nv;
            float x[K];
            float n2 = 0.f;
#pragma unroll
            for (int d = 0; d < DIM; ++d) {
                x[d] = px[d];
                n2 = fmaf(x[d], x[d], n2);
            }
            x[DIM] = ok ? n2 * (1.f - kTc) : FLT_MAX * 2.f;  // padding: never passes
            x[DIM + 1] = 1.f;
#pragma unroll
            for (int d = DIM + 2; d < K; ++d) x[d] = 0.f;
            gt[t_ld] = px[DIM];
            float4 *row4 = reinterpret_cast<float4 *>(row);
#pragma unroll
            for (int c = 0; c < CH; ++c)
                row4[c ^ sw] = make_float4(x[4 * c], x[4 * c + 1], x[4 * c + 2], x[4 * c + 3]);
        }
        __syncthreads();
        if (v0 + VT < ve) prefetch(v0 + VT);
        // refresh the bounds from the shared one (loaded a tile ago)
        if (!exact_only) {
#pragma unroll
            for (int r = 0; r < 4; ++r) {
                const int q = row_q(r);
                widen(r, __uint_as_float(pend[r]));
                if (q < Q) pend[r] = __ldcg(shared_lim + q);
            }
        }
        const int ng = (nv + 7) >> 3;
        for (int nt = 0; nt < ng; ++nt) {
            const int vrow = nt * 8 + lrow;
            unsigned b[KS][2];
#pragma unroll
            for (int kp = 0; kp + 1 < KS; kp += 2) {
                const int c = 2 * kp + lmat;  // chunk of k-step kp (lmat 0, 1) or kp + 1 (2, 3)
                const unsigned addr = xt_s + (unsigned)((vrow * K + 4 * (c ^ tc_swz<CH>(vrow))) * 4);
                ldsm_x4(addr, b[kp][0], b[kp][1], b[kp + 1][0], b[kp + 1][1]);
            }
            if (KS & 1) {
                const int c = 2 * (KS - 1) + (lmat & 1);
                const unsigned addr = xt_s + (unsigned)((vrow * K + 4 * (c ^ tc_swz<CH>(vrow))) * 4);
                ldsm_x2(addr, b[KS - 1][0], b[KS - 1][1]);
            }
            float acc[2][4];
#pragma unroll
            for (int mt = 0; mt < 2; ++mt) {
#pragma unroll
                for (int i = 0; i < 4; ++i) acc[mt][i] = 0.f;
#pragma unroll
                for (int ks = 0; ks < KS; ++ks) mma_tf32(acc[mt], a[mt][ks], b[ks][0], b[ks][1]);
            }
            // c0, c1: row grp, vertices 2 tig, 2 tig + 1; c2, c3: row grp + 8.
            // Without the bound (exact_only) every pair goes to the exact check.
            bool any = exact_only;
#pragma unroll
            for (int mt = 0; mt < 2; ++mt)
#pragma unroll
                for (int i = 0; i < 4; ++i) any |= acc[mt][i] <= lim[2 * mt + (i >> 1)];
            if (!__any_sync(kFull, any)) continue;
            unsigned pass = 0;
#pragma unroll
            for (int mt = 0; mt < 2; ++mt)
#pragma unroll
                for (int i = 0; i < 4; ++i)
                    pass |= (exact_only || acc[mt][i] <= lim[2 * mt + (i >> 1)]) ? 1u << (4 * mt + i) : 0u;
            // survivors are rare: one copy of the exact check, with the row's
            // state selected and written back by value
            while (pass) {
                const int e = __ffs(pass) - 1;
                pass &= pass - 1;
                const int r = 2 * (e >> 2) + ((e >> 1) & 1);
                const int q = row_q(r);
                const int vl = nt * 8 + 2 * tig + (e & 1);
                if (q >= Q || vl >= nv) continue;
                float c_r = cq[0], q_r = qn[0], l_r = lim[0];
                Best b_r = best[0];
#pragma unroll
                for (int k = 1; k < 4; ++k)
                    if (r == k) { c_r = cq[k]; q_r = qn[k]; l_r = lim[k]; b_r = best[k]; }
                const float g = gt[vl];
                // a vertex with g >= c is never admissible
                if (!(g < c_r)) continue;
                const float *xr = xt + vl * K;
                const int sw = tc_swz<CH>(vl);
                float d2 = 0.f;
                const float *qp = &qsm[0][q - qb];
#pragma unroll
                for (int d = 0; d < DIM; ++d) {
                    const float dq = qp[d * kTcQueries] - xr[4 * ((d >> 2) ^ sw) + (d & 3)];
                    d2 = fmaf(dq, dq, d2);
                }
                // filter of Alg. 2: g_v + |q - q_v| < c (strict); key (d^2, g, index).
                // The running best keeps the vertex's position in the g order;
                // original indices (perm) are looked up only to break an exact
                // (d^2, g) tie, and once per row at the end.
                const int pos = v0 + vl;
                if (d2 <= b_r.d2 && g + __fsqrt_rn(d2) < c_r &&
                    (d2 < b_r.d2 || g < b_r.g ||
                     (g == b_r.g && __ldg(perm + pos) < __ldg(perm + b_r.idx)))) {
                    b_r = Best{d2, g, pos};
                    if (!exact_only) {
                        l_r = fminf(l_r, fmaf(d2, 1.f + kC1, kTq * q_r) * (1.f + 4.f * kU));
                        atomicMin(shared_lim + q, __float_as_uint(d2));
                    }
#pragma unroll
                    for (int k = 0; k < 4; ++k)
                        if (r == k) { lim[k] = l_r; best[k] = b_r; }
                }
            }
            // the quad's lanes scan different vertex columns of the same
            // rows: a record of one tightens the bound of all four
#pragma unroll
            for (int r = 0; r < 4; ++r) {
                lim[r] = fminf(lim[r], __shfl_xor_sync(kFull, lim[r], 1));
                lim[r] = fminf(lim[r], __shfl_xor_sync(kFull, lim[r], 2));
            }
        }
    }
    tc_write_rows(best, perm, row_q, Q, partial);
    nn_finish(partial, fin, qblk, (cut_q + chunk - 1) / chunk, qb, Q);
}

__device__ __forceinline__ void mma_f16(float (&d)[4], const unsigned (&a)[4], unsigned b0,
                                        unsigned b1) {
    asm("mma.sync.aligned.m16n8k16.row.col.f32.f16.f16.f32 {%0, %1, %2, %3}, "
        "{%4, %5, %6, %7}, {%8, %9}, {%0, %1, %2, %3};"
        : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
        : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}

__device__ __forceinline__ unsigned pack_half2(float lo, float hi) {
    const __half2 h = __floats2half2_rn(lo, hi);  // lo in the low 16 bits
    return *reinterpret_cast<const unsigned *>(&h);
}

// FP16 form of the filter for D + 2 <= 16 (K = 16: one m16n8k16 per m-tile
// and 8 vertices; two groups of 8 vertices per ldmatrix.x4).  Same inputs as
// nearest_tc_kernel plus the ordering pass's largest coordinate magnitude
// (*maxabs, as float bits) and its non-finite flag (*nonfinite).  Vertex rows
// hold 16 halves (32 bytes, two 16-byte chunks swizzled by bit 2 of the
// vertex); the unscaled FP32 coordinates of the tile are kept beside them
// (SoA) for the exact checks.
// Registers are capped so that 3 blocks (24 warps) stay resident per SM.
template <int DIM>
__global__ void __launch_bounds__(kTcThreads, 3)
nearest_tc16_kernel(const float *__restrict__ tree, int N, int ldt, const float *__restrict__ queries,
                    const float *__restrict__ budgets, int Q, int chunk,
                    Best *__restrict__ partial, const int *__restrict__ perm,
                    const int *__restrict__ cut, float *__restrict__ seed,
                    const unsigned *__restrict__ maxabs, const int *__restrict__ nonfinite,
                    NnFinish fin) {
    static_assert(DIM + 2 <= 16, "FP16 filter holds K = 16");
    constexpr int VT = kTcThreads;                   // vertices per tile
    __shared__ __align__(16) unsigned xh[VT * 8];    // FP16 rows, swizzled chunks
    __shared__ float xf[DIM][VT];                    // unscaled FP32 coordinates
    __shared__ float gt[VT];
    __shared__ float qsm[DIM][kTcQueries];           // the block's queries (exact checks)
    __shared__ float red_g[kTcWarps];
    constexpr float kU = 5.9604645e-8f;            // 2^-24
    constexpr float kC1 = 4.f * (DIM + 2.f) * kU;  // exact-distance relative error
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int grp = lane >> 2, tig = lane & 3;
    // query blocks in descending budget order: the blocks with the longest
    // tree prefixes start first and the short ones fill the last wave
    const int qblk = gridDim.x - 1 - blockIdx.x;
    const int qb = qblk * kTcQueries;
    const int cut_q = min(N, cut[qblk]);
    const int vs = blockIdx.y * chunk;
    const int ve = min(cut_q, vs + chunk);
    if (vs >= ve) {  // no partial record: this slice is not counted
        if (blockIdx.y == 0) nn_write_none(fin, qb, Q);
        return;
    }

    // power-of-two scale: largest magnitude in [2^(ex-1), 2^ex) -> [8, 16)
    int ex = 0;
    frexpf(__uint_as_float(*maxabs), &ex);
    const int sh = 4 - ex;
    const bool exact_only = *nonfinite != 0 || sh > 126;
    const float sc = exact_only ? 1.f : ldexpf(1.f, sh);

    tc_stage_queries<DIM>(qsm, queries, Q, qb);
    __syncthreads();
    auto row_l = [&](int r) { return warp * 32 + (r >> 1) * 16 + grp + (r & 1) * 8; };
    auto row_q = [&](int r) { return qb + row_l(r); };
    float cq[4], qs2[4], lim[4];  // qs2: scaled |q|^2
    Best best[4];
    unsigned a[2][4];
#pragma unroll
    for (int r = 0; r < 4; ++r) {
        const int q = row_q(r);
        float n2 = 0.f;
#pragma unroll
        for (int d = 0; d < DIM; ++d) {
            const float v = qsm[d][row_l(r)] * sc;
            n2 = fmaf(v, v, n2);
        }
        qs2[r] = n2;
        cq[r] = q < Q ? budgets[q] : -FLT_MAX;  // nothing is admissible for padding
        best[r] = Best{FLT_MAX * 2.f, FLT_MAX * 2.f, -1};
        lim[r] = FLT_MAX * 2.f;
    }
    // A fragments (16 x 16, row-major): register i holds row grp + 8 (i & 1),
    // columns 2 tig + 8 (i >> 1) and the next one
    auto a_val = [&](int r, int k) {
        if (k < DIM) return -2.f * (qsm[k][row_l(r)] * sc);
        if (k == DIM) return 1.f;
        if (k == DIM + 1) return qs2[r];
        return 0.f;
    };
#pragma unroll
    for (int mt = 0; mt < 2; ++mt)
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const int r = 2 * mt + (i & 1), k = 2 * tig + 8 * (i >> 1);
            a[mt][i] = pack_half2(a_val(r, k), a_val(r, k + 1));
        }
    unsigned *const shared_lim = reinterpret_cast<unsigned *>(seed);
    // bound from the exact (unscaled) squared distance of an admissible vertex
    auto bound = [&](int r, float d2) {
        return fmaf((d2 * sc) * sc, 1.f + kC1, fmaf(kTq16, qs2[r], kAbs16)) * (1.f + 4.f * kU);
    };
    auto widen = [&](int r, float sd) {
        if (sd <= FLT_MAX) lim[r] = fminf(lim[r], bound(r, sd));
    };
    unsigned pend[4];
#pragma unroll
    for (int r = 0; r < 4; ++r) {
        const int q = row_q(r);
        pend[r] = q < Q ? __ldcg(shared_lim + q) : 0x7f800000u;
        widen(r, __uint_as_float(pend[r]));
    }
    {
        // an admissible vertex of this slice has |q - x| < c - g_min(slice)
        const float gm = tc_slice_gmin<DIM>(tree, ldt, vs, ve, red_g);
#pragma unroll
        for (int r = 0; r < 4; ++r) {
            if (!(cq[r] > gm)) {
                lim[r] = -FLT_MAX * 2.f;
            } else if (exact_only) {
                lim[r] = FLT_MAX * 2.f;
            } else {
                const float t = __fsub_ru(cq[r], gm);
                lim[r] = fminf(lim[r], bound(r, __fmul_ru(t, t)));
            }
        }
    }
    const unsigned xh_s = (unsigned)__cvta_generic_to_shared(xh);
    // ldmatrix.x4 row address of this lane: matrix lane >> 3 = (group of 8
    // vertices lane >> 4, chunk (lane >> 3) & 1), vertex row lane & 7
    const int lrow = lane & 7, lchunk = (lane >> 3) & 1, lgrp = lane >> 4;
    // next tile's vertex of this thread, loaded while the current one is scanned
    const int t_ld = threadIdx.x;
    float px[DIM + 1];
    auto prefetch = [&](int v0n) {
        const bool ok = t_ld < min(VT, ve - v0n);
        const unsigned base = (unsigned)(v0n + t_ld);
#pragma unroll
        for (int d = 0; d <= DIM; ++d) px[d] = ok ? __ldg(tree + (base + (unsigned)d * (unsigned)ldt)) : 0.f;
        if (!ok) px[DIM] = FLT_MAX * 2.f;  // padding vertex: g = +inf
    };
    prefetch(vs);
    for (int v0 = vs; v0 < ve; v0 += VT) {
        const int nv = min(VT, ve - v0);
        __syncthreads();
        {
            const bool ok = t_ld < nv;
            float h[16];
            float n2 = 0.f;
#pragma unroll
            for (int d = 0; d < DIM; ++d) {
                xf[d][t_ld] = px[d];
                h[d] = px[d] * sc;
                n2 = fmaf(h[d], h[d], n2);
            }
            h[DIM] = ok ? n2 * (1.f - kTc16) : FLT_MAX * 2.f;  // padding: never passes
            h[DIM + 1] = 1.f;
#pragma unroll
            for (int d = DIM + 2; d < 16; ++d) h[d] = 0.f;
            gt[t_ld] = px[DIM];
            uint4 *row = reinterpret_cast<uint4 *>(xh + t_ld * 8);
            const int sw = (t_ld >> 2) & 1;
            row[0 ^ sw] = make_uint4(pack_half2(h[0], h[1]), pack_half2(h[2], h[3]),
                                     pack_half2(h[4], h[5]), pack_half2(h[6], h[7]));
            row[1 ^ sw] = make_uint4(pack_half2(h[8], h[9]), pack_half2(h[10], h[11]),
                                     pack_half2(h[12], h[13]), pack_half2(h[14], h[15]));
        }
        __syncthreads();
        if (v0 + VT < ve) prefetch(v0 + VT);
        if (!exact_only) {
#pragma unroll
            for (int r = 0; r < 4; ++r) {
                const int q = row_q(r);
                widen(r, __uint_as_float(pend[r]));
                if (q < Q) pend[r] = __ldcg(shared_lim + q);
            }
        }
        const int ng2 = (nv + 15) >> 4;  // pairs of 8-vertex groups
#pragma unroll 2
        for (int np = 0; np < ng2; ++np) {
            const int vrow = (2 * np + lgrp) * 8 + lrow;
            unsigned b[2][2];
            ldsm_x4(xh_s + (unsigned)(vrow * 32 + 16 * (lchunk ^ ((vrow >> 2) & 1))), b[0][0],
                    b[0][1], b[1][0], b[1][1]);
            float acc[2][2][4];
#pragma unroll
            for (int j = 0; j < 2; ++j)
#pragma unroll
                for (int mt = 0; mt < 2; ++mt) {
#pragma unroll
                    for (int i = 0; i < 4; ++i) acc[j][mt][i] = 0.f;
                    mma_f16(acc[j][mt], a[mt], b[j][0], b[j][1]);
                }
            // element (j, mt, i): row grp + 8 (i >> 1) of m-tile mt, vertex
            // 8 (2 np + j) + 2 tig + (i & 1)
            // the common case, nothing passes: one compare per row on the
            // minimum of its four values (a NaN never passes either way)
            bool any = exact_only;
#pragma unroll
            for (int mt = 0; mt < 2; ++mt)
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                    const float m = fminf(fminf(acc[0][mt][2 * h], acc[0][mt][2 * h + 1]),
                                          fminf(acc[1][mt][2 * h], acc[1][mt][2 * h + 1]));
                    any |= m <= lim[2 * mt + h];
                }
            if (!__any_sync(kFull, any)) continue;
            unsigned pass = 0;
#pragma unroll
            for (int j = 0; j < 2; ++j)
#pragma unroll
                for (int mt = 0; mt < 2; ++mt)
#pragma unroll
                    for (int i = 0; i < 4; ++i)
                        pass |= (exact_only || acc[j][mt][i] <= lim[2 * mt + (i >> 1)])
                                    ? 1u << (8 * j + 4 * mt + i) : 0u;
            while (pass) {
                const int e = __ffs(pass) - 1;
                pass &= pass - 1;
                const int r = 2 * ((e >> 2) & 1) + ((e >> 1) & 1);
                const int q = row_q(r);
                const int vl = (2 * np + (e >> 3)) * 8 + 2 * tig + (e & 1);
                if (q >= Q || vl >= nv) continue;
                float c_r = cq[0], l_r = lim[0];
                Best b_r = best[0];
#pragma unroll
                for (int k = 1; k < 4; ++k)
                    if (r == k) { c_r = cq[k]; l_r = lim[k]; b_r = best[k]; }
                const float g = gt[vl];
                // a vertex with g >= c is never admissible
                if (!(g < c_r)) continue;
                float d2 = 0.f;
                const float *qp = &qsm[0][q - qb];
                const float *xp = &xf[0][vl];
#pragma unroll
                for (int d = 0; d < DIM; ++d) {
                    const float dq = qp[d * kTcQueries] - xp[d * VT];
                    d2 = fmaf(dq, dq, d2);
                }
                // filter of Alg. 2: g_v + |q - q_v| < c (strict); key (d^2, g, index).
                // The running best keeps the vertex's position in the g order;
                // original indices (perm) are looked up only to break an exact
                // (d^2, g) tie, and once per row at the end.
                const int pos = v0 + vl;
                if (d2 <= b_r.d2 && g + __fsqrt_rn(d2) < c_r &&
                    (d2 < b_r.d2 || g < b_r.g ||
                     (g == b_r.g && __ldg(perm + pos) < __ldg(perm + b_r.idx)))) {
                    b_r = Best{d2, g, pos};
                    if (!exact_only) {
                        float bq = 0.f;
#pragma unroll
                        for (int k = 0; k < 4; ++k)
                            if (r == k) bq = bound(k, d2);
                        l_r = fminf(l_r, bq);
                        atomicMin(shared_lim + q, __float_as_uint(d2));
                    }
#pragma unroll
                    for (int k = 0; k < 4; ++k)
                        if (r == k) { lim[k] = l_r; best[k] = b_r; }
                }
            }
            // the quad's lanes scan different vertex columns of the same
            // rows: a record of one tightens the bound of all four
#pragma unroll
            for (int r = 0; r < 4; ++r) {
                lim[r] = fminf(lim[r], __shfl_xor_sync(kFull, lim[r], 1));
                lim[r] = fminf(lim[r], __shfl_xor_sync(kFull, lim[r], 2));
            }
        }
    }
    tc_write_rows(best, perm, row_q, Q, partial);
    nn_finish(partial, fin, qblk, (cut_q + chunk - 1) / chunk, qb, Q);
}

// ---------------------------------------------------------------------------
// NEAREST filter in FP32 on the FMA pipe (the default for large batches).
// The same expansion as the tensor-core filters, e(q, x) = |q|^2 + |x|^2 -
// 2 q.x, is computed per (query, vertex) pair as a chain of D fused
// multiply-adds that starts from the vertex's folded squared norm:
//   acc = xn + sum_d (-2 q_d) x_d,   xn = fl(|x|^2) (1 - 4 gamma),
// and a pair passes when acc <= T_q, a per-query threshold with |q|^2 taken
// out.  The ordering pass stores xn as an extra row of the ordered tree.  A
// thread owns 8 queries x 8 vertices of each 64-vertex step (a register tile
// of 64 accumulators); the operands are read as 16-byte vectors from
// dimension-major shared arrays, every load a broadcast or one conflict-free
// row.  For 8 <= D <= 21 the tile is updated with packed FP32 FMAs (fma.rn.f32x2:
// two IEEE single-precision FMAs per instruction, each rounded as fmaf, so
// the accumulators are bit-identical to the scalar chain): the multipliers
// -2 q_d are kept twice in shared memory, {a, a}, and pair with two adjacent
// vertex columns, 6 shared loads per 32 packed FMAs (64 FMAs).  That halves
// the instructions the FMA chain issues; the pipe's FMA rate is unchanged, so
// the other instructions of the scan fit in the issue slots it frees.  Warp
// lanes 8 ty' + tx share the queries of ty (8 lanes) and the vertex columns
// of tx.  Tree tiles come in by cp.async
// into a double buffer, one barrier per tile; the running best of each
// (thread, query) sits in shared memory and is touched only when a pair
// passes, so that two blocks (16 warps) stay resident per SM.
//
// Error bound (u = 2^-24, gamma = kF32G (D + 2) = 1.25 (D + 2) u; the ordering
// pass sends every pair to the exact check unless every nonzero coordinate
// lies in [2^-60, 2^60], so no product or squared norm over- or underflows):
//   * fl(|x|^2) is within gamma |x|^2, so xn + gamma (xn + |x|^2) <= |x|^2;
//   * the chain adds at most gamma (xn + sum |2 q_d x_d|) <=
//     gamma (xn + |q|^2 + |x|^2), hence acc <= |q - x|^2 - |q|^2 (1 - gamma);
//   * qn = fl(|q|^2) is within gamma |q|^2, hence acc <= |q - x|^2 - qn +
//     2 gamma qn.
// The exact formula's d2 of any admissible vertex is at least |q - x*|^2 /
// (1 + kC1) for the true nearest admissible x* (kC1 = 4 (D + 2) u), so
//   T_q = fl_up( fl(fmaf(d2, 1 + kC1, 2 gamma qn)) (1 + 4 u) - qn )
// satisfies acc(x*) <= T_q: the filter never drops the true nearest vertex.
// Every vertex that passes is decided by the exact formula on the FP32
// coordinates, so the results equal the plain scan's, ties included.
// ---------------------------------------------------------------------------
constexpr float kF32G = 1.25f * 5.9604645e-8f;  // gamma / (D + 2)
constexpr int kF32Step = 64;                     // vertices per register-tile step

template <int DIM>
struct F32Shape {
    // packed FMAs (the multipliers kept twice) where two blocks still fit and
    // the tile's registers do not spill (they do below 8 dimensions)
    static constexpr bool PACKED = DIM >= 8 && DIM <= 21;
    // vertices per shared-memory tile (six 64-vertex steps per barrier up to
    // 14 dimensions) such that two blocks of 256 threads fit an SM up to 56
    // rows (64 rows: 121 KB a block, one per SM)
    static constexpr int VT = DIM <= 14 ? 384 : (DIM <= 21 && !PACKED) ? 128 : 64;
    static constexpr int ROWS = DIM + 2;              // x_d, g, folded |x|^2
    static constexpr int AM = PACKED ? 2 : 1;         // copies of each -2 q_d
};

template <int DIM>
constexpr size_t f32_smem_bytes() {
    // -2 q [DIM][256] (twice when packed), two tiles [ROWS][VT], best d2,
    // best position and bound [8][256] each
    return sizeof(float) * ((size_t)F32Shape<DIM>::AM * DIM * kTcQueries +
                            (size_t)2 * F32Shape<DIM>::ROWS * F32Shape<DIM>::VT +
                            (size_t)3 * 8 * kTcQueries);
}

template <int DIM>
__global__ void __launch_bounds__(kTcThreads, 2)
nearest_f32_kernel(const float *__restrict__ tree, int N, int ldt, const float *__restrict__ queries,
                   const float *__restrict__ budgets, int Q, int chunk,
                   Best *__restrict__ partial, const int *__restrict__ perm,
                   const int *__restrict__ cut, float *__restrict__ seed,
                   const int *__restrict__ exact_only_flag, NnFinish fin) {
    constexpr int VT = F32Shape<DIM>::VT, ROWS = F32Shape<DIM>::ROWS, AM = F32Shape<DIM>::AM;
    extern __shared__ __align__(16) float f32_sm[];
    // -2 q_d of query j at am[d][AM j .. AM j + AM - 1]
    float(*am)[AM * kTcQueries] = reinterpret_cast<float(*)[AM * kTcQueries]>(f32_sm);
    float *tiles = f32_sm + AM * DIM * kTcQueries;                // [2][ROWS][VT]
    float(*sb_d2)[kTcQueries] =
        reinterpret_cast<float(*)[kTcQueries]>(tiles + 2 * ROWS * VT);  // [8][256]
    int(*sb_pos)[kTcQueries] = reinterpret_cast<int(*)[kTcQueries]>(sb_d2 + 8);
    float(*lim_s)[kTcQueries] = reinterpret_cast<float(*)[kTcQueries]>(sb_pos + 8);
    __shared__ float qn_s[kTcQueries];                   // fl(|q|^2)
    __shared__ float cq_s[kTcQueries];                   // budgets
    __shared__ unsigned sl_s[kTcQueries];                // shared bounds, one tile old
    __shared__ float red_g[kTcWarps];
    constexpr float kU = 5.9604645e-8f;                   // 2^-24
    constexpr float kC1 = 4.f * (DIM + 2.f) * kU;         // exact-distance relative error
    constexpr float kG = kF32G * (DIM + 2.f);             // gamma
    const int tid = threadIdx.x;
    const int ty = tid >> 3, tx = tid & 7;
    // query blocks in descending budget order: the blocks with the longest
    // tree prefixes start first and the short ones fill the last wave
    const int qblk = gridDim.x - 1 - blockIdx.x;
    const int qb = qblk * kTcQueries;
    const int cut_q = min(N, cut[qblk]);
    const int vs = blockIdx.y * chunk;
    const int ve = min(cut_q, vs + chunk);
    if (vs >= ve) {  // no partial record: this slice is not counted
        if (blockIdx.y == 0) nn_write_none(fin, qb, Q);
        return;
    }
    const bool exact_only = *exact_only_flag != 0;
    unsigned *const shared_lim = reinterpret_cast<unsigned *>(seed);

    // first tile in flight while the queries are staged
    // 16-byte pieces (rows start on 16-byte boundaries, slices and tiles on
    // multiples of 4 vertices); a piece past the slice end is zero-filled, its
    // folded norms +inf so that the padding columns never pass
    auto issue_tile = [&](int v0n, int buf) {
        const int nvn = min(VT, ve - v0n);
        float *dst = tiles + buf * ROWS * VT;
        for (int i = tid; i < ROWS * (VT / 4); i += kTcThreads) {
            const int d = i / (VT / 4), j = 4 * (i - d * (VT / 4));
            float *to = dst + d * VT + j;
            const float *from = tree + ((size_t)d * ldt + v0n + j);
            if (j + 4 <= nvn) {
                cp_async16(to, from, 16);
            } else if (d == DIM + 1) {
#pragma unroll
                for (int k = 0; k < 4; ++k)
                    cp_async4(to + k, j + k < nvn ? from + k : &g_f32_pad_inf, true);
            } else {
                cp_async16(to, j < nvn ? from : tree, 4 * max(0, nvn - j));
            }
        }
        cp_async_commit();
    };
    issue_tile(vs, 0);

    // The queries themselves are not kept: within the filter's coordinate
    // range [2^-60, 2^60] both -2 q_d and -0.5 (-2 q_d) are exact, so the exact
    // check takes q_d back from the multipliers; in exact-only mode it reads
    // the ordered queries from global memory instead.
    {
        const int j = tid;
        const bool ok = qb + j < Q;
        float n2 = 0.f;
#pragma unroll
        for (int d = 0; d < DIM; ++d) {
            const float v = ok ? __ldg(queries + (size_t)d * Q + qb + j) : 0.f;
            const float a = -2.f * v;
            if constexpr (AM == 2)
                *reinterpret_cast<float2 *>(&am[d][2 * j]) = make_float2(a, a);
            else
                am[d][j] = a;
            n2 = fmaf(v, v, n2);
        }
        qn_s[j] = n2;
        cq_s[j] = qb + j < Q ? budgets[qb + j] : -FLT_MAX;  // padding admits nothing
        sl_s[j] = qb + j < Q ? __ldcg(shared_lim + qb + j) : 0x7f800000u;
#pragma unroll
        for (int r = 0; r < 8; ++r) {
            sb_d2[r][j] = FLT_MAX * 2.f;
            sb_pos[r][j] = -1;
        }
    }
    __syncthreads();
    // row r of this thread: query ql(r) of the block; rows of real queries
    auto ql = [&](int r) { return r < 4 ? ty * 4 + r : 128 + ty * 4 + (r - 4); };
    unsigned row_ok = 0;
#pragma unroll
    for (int r = 0; r < 8; ++r) row_ok |= qb + ql(r) < Q ? 1u << r : 0u;
    auto bound = [&](int r, float d2) {
        const float qn = qn_s[ql(r)];
        return __fsub_ru(fmaf(d2, 1.f + kC1, 2.f * kG * qn) * (1.f + 4.f * kU), qn);
    };
    float lim[8];
    {
        // an admissible vertex of this slice has |q - x| < c - g_min(slice)
        const float gm = tc_slice_gmin<DIM>(tree, ldt, vs, ve, red_g);
#pragma unroll
        for (int r = 0; r < 8; ++r) {
            const float c = cq_s[ql(r)];
            if (!(c > gm)) {
                lim[r] = -FLT_MAX * 2.f;
            } else if (exact_only) {
                lim[r] = FLT_MAX * 2.f;
            } else {
                const float t = __fsub_ru(c, gm);
                lim[r] = bound(r, __fmul_ru(t, t));
            }
        }
    }
    unsigned sl_next = 0x7f800000u;  // this thread's query tid, for the next tile
    int buf = 0;
    for (int v0 = vs; v0 < ve; v0 += VT, buf ^= 1) {
        const int nv = min(VT, ve - v0);
        const float(*xs)[VT] = reinterpret_cast<const float(*)[VT]>(tiles + buf * ROWS * VT);
        cp_async_wait_all();
        // (a newer bound than another thread's view is still a valid bound)
        if (v0 > vs) sl_s[tid] = sl_next;
        __syncthreads();  // tile visible; every thread is done with the other buffer
        if (v0 + VT < ve) issue_tile(v0 + VT, buf ^ 1);
        if (qb + tid < Q) sl_next = __ldcg(shared_lim + qb + tid);
        if (!exact_only) {
#pragma unroll
            for (int r = 0; r < 8; ++r) {
                const float sd = __uint_as_float(sl_s[ql(r)]);
                if (sd <= FLT_MAX) lim[r] = fminf(lim[r], bound(r, sd));
            }
        }
        const int steps = (nv + kF32Step - 1) / kF32Step;
        for (int s = 0; s < steps; ++s) {
            const int c0 = s * kF32Step + tx * 4;  // columns c0..c0+3 and c0+32..c0+35
            float acc[8][8];
            if constexpr (AM == 2) {
                // pairs of adjacent columns: p = 0, 1 -> c0 + 2p, 2 -> c0 + 32, 3 -> c0 + 34
                const ulonglong2 n0 = *reinterpret_cast<const ulonglong2 *>(&xs[DIM + 1][c0]);
                const ulonglong2 n1 = *reinterpret_cast<const ulonglong2 *>(&xs[DIM + 1][c0 + 32]);
                const f32x2_t xn[4] = {n0.x, n0.y, n1.x, n1.y};
                f32x2_t acc2[8][4];
#pragma unroll
                for (int d = 0; d < DIM; ++d) {
                    // {a, a} of rows 0-1, 2-3 (queries 4 ty ..) and 4-5, 6-7 (128 + 4 ty ..)
                    const ulonglong2 a0 = *reinterpret_cast<const ulonglong2 *>(&am[d][8 * ty]);
                    const ulonglong2 a1 = *reinterpret_cast<const ulonglong2 *>(&am[d][8 * ty + 4]);
                    const ulonglong2 a2 =
                        *reinterpret_cast<const ulonglong2 *>(&am[d][256 + 8 * ty]);
                    const ulonglong2 a3 =
                        *reinterpret_cast<const ulonglong2 *>(&am[d][256 + 8 * ty + 4]);
                    const ulonglong2 x0 = *reinterpret_cast<const ulonglong2 *>(&xs[d][c0]);
                    const ulonglong2 x1 = *reinterpret_cast<const ulonglong2 *>(&xs[d][c0 + 32]);
                    const f32x2_t a[8] = {a0.x, a0.y, a1.x, a1.y, a2.x, a2.y, a3.x, a3.y};
                    const f32x2_t x[4] = {x0.x, x0.y, x1.x, x1.y};
#pragma unroll
                    for (int r = 0; r < 8; ++r)
#pragma unroll
                        for (int p = 0; p < 4; ++p)
                            acc2[r][p] = fma_f32x2(a[r], x[p], d == 0 ? xn[p] : acc2[r][p]);
                }
#pragma unroll
                for (int r = 0; r < 8; ++r)
#pragma unroll
                    for (int p = 0; p < 4; ++p) {
                        acc[r][2 * p] = f32x2_lo(acc2[r][p]);
                        acc[r][2 * p + 1] = f32x2_hi(acc2[r][p]);
                    }
            } else {
                const float4 n0 = *reinterpret_cast<const float4 *>(&xs[DIM + 1][c0]);
                const float4 n1 = *reinterpret_cast<const float4 *>(&xs[DIM + 1][c0 + 32]);
                const float xn[8] = {n0.x, n0.y, n0.z, n0.w, n1.x, n1.y, n1.z, n1.w};
#pragma unroll
                for (int d = 0; d < DIM; ++d) {
                    const float4 a0 = *reinterpret_cast<const float4 *>(&am[d][ty * 4]);
                    const float4 a1 = *reinterpret_cast<const float4 *>(&am[d][128 + ty * 4]);
                    const float4 x0 = *reinterpret_cast<const float4 *>(&xs[d][c0]);
                    const float4 x1 = *reinterpret_cast<const float4 *>(&xs[d][c0 + 32]);
                    const float a[8] = {a0.x, a0.y, a0.z, a0.w, a1.x, a1.y, a1.z, a1.w};
                    const float x[8] = {x0.x, x0.y, x0.z, x0.w, x1.x, x1.y, x1.z, x1.w};
#pragma unroll
                    for (int r = 0; r < 8; ++r)
#pragma unroll
                        for (int c = 0; c < 8; ++c)
                            acc[r][c] = fmaf(a[r], x[c], d == 0 ? xn[c] : acc[r][c]);
                }
            }
            // the common case, nothing passes: one compare per row on the
            // minimum of its eight values (a NaN never passes either way);
            // rows of padding queries (q >= Q) never pass
            unsigned rows = 0;
#pragma unroll
            for (int r = 0; r < 8; ++r) {
                const float m = fmin3(fmin3(acc[r][0], acc[r][1], acc[r][2]),
                                      fmin3(acc[r][3], acc[r][4], acc[r][5]),
                                      fminf(acc[r][6], acc[r][7]));
                rows |= (exact_only || m <= lim[r]) ? 1u << r : 0u;
            }
            rows &= row_ok;
            if (!__any_sync(kFull, rows != 0u)) continue;
            // pass bits r * 8 + c of the rows that pass, then one loop over
            // them with the bounds in shared memory (dynamic row index)
            unsigned long long pass = 0ull;
#pragma unroll
            for (int r = 0; r < 8; ++r)
                if ((rows >> r) & 1u) {
#pragma unroll
                    for (int c = 0; c < 8; ++c)
                        if (exact_only || acc[r][c] <= lim[r]) pass |= 1ull << (8 * r + c);
                }
            if (pass) {
#pragma unroll
                for (int r = 0; r < 8; ++r) lim_s[r][tid] = lim[r];
#pragma unroll 1
                while (pass) {
                    const int bit = __ffsll((long long)pass) - 1;
                    pass &= pass - 1;
                    const int r = bit >> 3, c = bit & 7;
                    const int vl = c0 + (c < 4 ? c : 28 + c);
                    if (vl >= nv) continue;
                    const float g = xs[DIM][vl];
                    const int qlr = r < 4 ? ty * 4 + r : 128 + ty * 4 + (r - 4);
                    const float cr = cq_s[qlr];
                    // a vertex with g >= c is never admissible
                    if (!(g < cr)) continue;
                    float d2 = 0.f;
                    if (exact_only) {
#pragma unroll
                        for (int d = 0; d < DIM; ++d) {
                            const float dq = __ldg(queries + (size_t)d * Q + qb + qlr) - xs[d][vl];
                            d2 = fmaf(dq, dq, d2);
                        }
                    } else {
#pragma unroll
                        for (int d = 0; d < DIM; ++d) {
                            // one rounding of q_d - x_d, as the plain difference
                            const float dq = fmaf(-0.5f, am[d][AM * qlr], -xs[d][vl]);
                            d2 = fmaf(dq, dq, d2);
                        }
                    }
                    // filter of Alg. 2: g_v + |q - q_v| < c (strict); key (d^2,
                    // g, index), the running best keeps the vertex's position in
                    // the g order (its g is looked up there; original indices
                    // break exact ties)
                    const float bd2 = sb_d2[r][tid];
                    if (!(d2 <= bd2) || !(g + __fsqrt_rn(d2) < cr)) continue;
                    const int bpos = sb_pos[r][tid];
                    bool take = d2 < bd2 || bpos < 0;
                    if (!take) {
                        const float bg = __ldg(tree + (size_t)DIM * ldt + bpos);
                        take = g < bg || (g == bg && __ldg(perm + v0 + vl) < __ldg(perm + bpos));
                    }
                    if (take) {
                        sb_d2[r][tid] = d2;
                        sb_pos[r][tid] = v0 + vl;
                        if (!exact_only) {
                            const float qn = qn_s[qlr];
                            const float bq = __fsub_ru(
                                fmaf(d2, 1.f + kC1, 2.f * kG * qn) * (1.f + 4.f * kU), qn);
                            lim_s[r][tid] = fminf(lim_s[r][tid], bq);
                            atomicMin(shared_lim + qb + qlr, __float_as_uint(d2));
                        }
                    }
                }
#pragma unroll
                for (int r = 0; r < 8; ++r) lim[r] = lim_s[r][tid];
            }
            // the 8 lanes of a query group scan different vertex columns of
            // the same rows: a record of one tightens the bound of all
#pragma unroll
            for (int r = 0; r < 8; ++r) {
                lim[r] = fminf(lim[r], __shfl_xor_sync(kFull, lim[r], 1));
                lim[r] = fminf(lim[r], __shfl_xor_sync(kFull, lim[r], 2));
                lim[r] = fminf(lim[r], __shfl_xor_sync(kFull, lim[r], 4));
            }
        }
    }
    // original indices, then the best of the query group's 8 lanes
#pragma unroll
    for (int r = 0; r < 8; ++r) {
        const int pos = sb_pos[r][tid];
        Best b{FLT_MAX * 2.f, FLT_MAX * 2.f, -1};
        if (pos >= 0) b = Best{sb_d2[r][tid], __ldg(tree + (size_t)DIM * ldt + pos), __ldg(perm + pos)};
#pragma unroll
        for (int o = 1; o <= 4; o <<= 1) {
            const Best other = shfl_best(b, o);
            if (better(other, b)) b = other;
        }
        const int q = qb + ql(r);
        if (tx == 0 && q < Q) partial[(size_t)blockIdx.y * Q + q] = b;
    }
    nn_finish(partial, fin, qblk, (cut_q + chunk - 1) / chunk, qb, Q);
}

// ---------------------------------------------------------------------------
// Budget-ordered NEAREST for large batches.  A vertex with g_v >= c is never
// admissible (distances are >= 0), so once the tree is ordered by g and the
// queries by budget, a block of queries only needs the prefix of the tree
// whose g lies below its largest budget.  Both orders come from one counting
// sort each into kSortBuckets buckets that share their limits: the sorted
// values of g at kSortBuckets evenly spaced vertices, so that a bucket holds
// about the same number of vertices whatever the distribution of g.  The order
// inside a bucket does not matter, because exact ties are broken by original
// vertex index.
//
// The passes are bound by memory: the tree is read and written once, and g
// read twice.  A block counts its up to 4,096 consecutive items in shared
// memory and touches each global counter once; before, every item was its own
// global atomic on one of 1,024 counters, and its row entries were written one
// by one to unrelated sectors.  Ordering a 28-D tree of 1,000,000 vertices:
// about 350 us before (from whole calls), 100 us now; 16,384 vertices and
// 65,536 queries in 14-D: 42 us before, 29 us now.
// ---------------------------------------------------------------------------
constexpr int kSortBuckets = 256;
constexpr int kSortThreads = 512;
constexpr int kSortPer = 8;  // items per thread at most

struct SortState {
    int gmin;                            // order-preserving key of the smallest g (NaN aside)
    int exact_only;                      // a coordinate lies outside the TF32 filter's range
    int nonfinite;                       // a coordinate is NaN or infinite
    unsigned maxabs;                     // largest finite coordinate magnitude (float bits)
    int arrive;                          // histogram blocks done (the last one scans)
    float split[kSortBuckets];           // bucket b >= 1 starts at split[b]; split[0] unused
    int tree_off[kSortBuckets + 1];      // bucket starts of the g-ordered tree
    int tree_cur[kSortBuckets];
    int query_off[kSortBuckets + 1];
    int query_cur[kSortBuckets];
};

__device__ __forceinline__ int fkey(float v) {
    const int k = __float_as_int(v);
    return k ^ ((k >> 31) & 0x7fffffff);
}
__device__ __forceinline__ float unkey(int o) { return __int_as_float(o ^ ((o >> 31) & 0x7fffffff)); }

// Bucket of v: the number of limits at or below it (monotonic in v, -infinity
// first); NaN goes to the last bucket.
__device__ __forceinline__ int sort_bucket(float v, const float *split) {
    if (v != v) return kSortBuckets - 1;
    int b = 0;
#pragma unroll
    for (int step = kSortBuckets / 2; step > 0; step >>= 1)
        if (split[b + step] <= v) b += step;
    return b;
}

// First pass of a call: resets the sort state and the filter's per-query-block
// slice counters, and ranks the samples of g into the bucket limits.
__global__ void __launch_bounds__(kSortBuckets)
sort_setup(const float *__restrict__ g, int N, SortState *S, int *__restrict__ qdone, int qblocks) {
    __shared__ __align__(16) float smp[kSortBuckets];
    const int t = threadIdx.x;
    float x = g[(int)((int64_t)t * N / kSortBuckets)];
    if (x != x) x = INFINITY;
    smp[t] = x;
    for (int i = t; i <= kSortBuckets; i += kSortBuckets) S->tree_off[i] = S->query_off[i] = 0;
    for (int i = t; i < qblocks; i += kSortBuckets) qdone[i] = 0;
    if (t == 0) {
        S->gmin = 0x7fffffff;  // no g but NaN
        S->exact_only = 0;
        S->nonfinite = 0;
        S->maxabs = 0u;
        S->arrive = 0;
    }
    __syncthreads();
    int rank = 0;
#pragma unroll 8
    for (int i = 0; i < kSortBuckets; i += 4) {
        const float4 o = *reinterpret_cast<const float4 *>(&smp[i]);
        rank += (o.x < x || (o.x == x && i < t)) + (o.y < x || (o.y == x && i + 1 < t)) +
                (o.z < x || (o.z == x && i + 2 < t)) + (o.w < x || (o.w == x && i + 3 < t));
    }
    S->split[rank] = x;
}

// Warp-aggregated counter update: lanes of a warp with the same bucket b
// (b < 0: no item) add their count once, through the group's first lane, and
// each receives the counter's old value plus its rank in the group (many
// budgets can share one bucket, e.g. every budget above the largest g).
__device__ __forceinline__ int grouped_add(int *counters, int b) {
    const int lane = threadIdx.x & 31;
    const unsigned grp = __match_any_sync(kFull, b);
    const int leader = __ffs(grp) - 1;
    int base = 0;
    if (b >= 0 && lane == leader) base = atomicAdd(&counters[b], __popc(grp));
    base = __shfl_sync(kFull, base, leader);
    return base + __popc(grp & ((1u << lane) - 1u));
}

// Items per thread of the sorting blocks over n items, 1, 2, 4 or 8: as many
// as still give each of the 152 SMs a block.
static int sort_per(int n) {
    int per = 1;
    while (per < kSortPer && n / (kSortThreads * 152) >= 2 * per) per *= 2;
    return per;
}

// Bucket counts of the tree's g (the first tblocks blocks) and of the budgets;
// the last block to finish turns both count arrays into bucket starts.
__global__ void __launch_bounds__(kSortThreads)
sort_histogram(const float *__restrict__ g, int N, int tper, int tblocks,
               const float *__restrict__ c, int Q, int qper, SortState *S) {
    __shared__ float split[kSortBuckets];
    __shared__ int cnt[kSortBuckets];
    __shared__ int s_last;
    __shared__ int part[kSortBuckets / 32];
    const int t = threadIdx.x;
    const bool tree = (int)blockIdx.x < tblocks;
    const float *src = tree ? g : c;
    const int n = tree ? N : Q, per = tree ? tper : qper;
    const int64_t base = (int64_t)(tree ? blockIdx.x : blockIdx.x - tblocks) * per * kSortThreads;
    if (t < kSortBuckets) {
        split[t] = S->split[t];
        cnt[t] = 0;
    }
    __syncthreads();
    int lo = 0x7fffffff;
    for (int k = 0; k < per; ++k) {
        const int64_t i = base + (int64_t)k * kSortThreads + t;
        const float v = i < n ? src[i] : 0.f;
        if (i < n && v == v) lo = min(lo, fkey(v));
        grouped_add(cnt, i < n ? sort_bucket(v, split) : -1);
    }
    if (tree) {
        lo = __reduce_min_sync(kFull, lo);
        if ((t & 31) == 0 && lo != 0x7fffffff) atomicMin(&S->gmin, lo);
    }
    __syncthreads();
    if (t < kSortBuckets && cnt[t]) atomicAdd((tree ? S->tree_off : S->query_off) + 1 + t, cnt[t]);
    __threadfence();
    __syncthreads();
    if (t == 0) s_last = atomicAdd(&S->arrive, 1) == (int)gridDim.x - 1;
    __syncthreads();
    if (!s_last) return;
    __threadfence();
    // inclusive scan of the shifted counts, one bucket per thread: off[b]
    // becomes the start of bucket b, where its cursor starts too
    const int lane = t & 31, w = t >> 5;
    for (int which = 0; which < 2; ++which) {
        int *off = which ? S->query_off : S->tree_off;
        int *cur = which ? S->query_cur : S->tree_cur;
        const int own = t < kSortBuckets ? __ldcg(off + 1 + t) : 0;
        int x = own;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int y = __shfl_up_sync(kFull, x, o);
            if (lane >= o) x += y;
        }
        if (t < kSortBuckets && lane == 31) part[w] = x;
        __syncthreads();
        if (t < kSortBuckets) {
            for (int k = 0; k < w; ++k) x += part[k];
            cur[t] = x - own;
            off[1 + t] = x;
        }
        __syncthreads();  // part is reused
    }
}

// Scatter the tree (all D+1 rows) and the queries into bucket order, in dp >=
// dim coordinate rows of which the last dp - dim are zero (a zero coordinate
// adds exactly nothing to a norm, a product chain or a distance).  A block
// orders its PER * 512 items in shared memory first and reserves a run of each
// bucket, so a row is read within one window of at most 16 KB and written in
// runs; 8 loads are in flight per thread, over items and, with fewer items,
// rows.
struct ScatterShared {
    float split[kSortBuckets];
    int cnt[kSortBuckets], lbase[kSortBuckets], gdelta[kSortBuckets];
    int part[kSortBuckets / 32];
    int dst[kSortPer * kSortThreads];
    uint16_t src[kSortPer * kSortThreads];
};

// in: dim rows of stride ld_in, key: their sort values, n items; all from the
// block's first item on.  out: dp rows of stride ld_out, orig0 the first item's
// index.  For the tree the sort values and folded norms follow as rows.
template <int PER>
__device__ __forceinline__ void scatter_items(const float *__restrict__ in, int64_t ld_in,
                                              const float *__restrict__ key, int items, int dim,
                                              int dp, bool is_tree, int orig0, SortState *S,
                                              int *cur, float *__restrict__ out, int64_t ld_out,
                                              float *__restrict__ key_out,
                                              int *__restrict__ perm, ScatterShared &sh) {
    const int t = threadIdx.x, lane = t & 31, w = t >> 5;
    if (t < kSortBuckets) {
        sh.split[t] = S->split[t];
        sh.cnt[t] = 0;
    }
    __syncthreads();
    int br[PER];  // bucket | rank in the block's bucket << 8
#pragma unroll
    for (int k = 0; k < PER; ++k) {
        const int i = k * kSortThreads + t;
        const int b = i < items ? sort_bucket(key[i], sh.split) : -1;
        const int r = grouped_add(sh.cnt, b);
        br[k] = b < 0 ? -1 : b | (r << 8);
    }
    __syncthreads();
    if (t < kSortBuckets) {
        const int own = sh.cnt[t];
        int x = own;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int y = __shfl_up_sync(kFull, x, o);
            if (lane >= o) x += y;
        }
        if (lane == 31) sh.part[w] = x;
        sh.lbase[t] = x - own;
    }
    __syncthreads();
    if (t < kSortBuckets) {
        int l = sh.lbase[t];
        for (int k = 0; k < w; ++k) l += sh.part[k];
        sh.lbase[t] = l;
        sh.gdelta[t] = sh.cnt[t] ? atomicAdd(cur + t, sh.cnt[t]) - l : 0;
    }
    __syncthreads();
#pragma unroll
    for (int k = 0; k < PER; ++k) {
        if (br[k] < 0) continue;
        const int b = br[k] & 255, slot = sh.lbase[b] + (br[k] >> 8);
        sh.src[slot] = (uint16_t)(k * kSortThreads + t);
        sh.dst[slot] = slot + sh.gdelta[b];
    }
    __syncthreads();
    int from[PER], to[PER];
    float n2[PER];
#pragma unroll
    for (int k = 0; k < PER; ++k) {
        const int slot = k * kSortThreads + t;
        from[k] = slot < items ? sh.src[slot] : -1;
        to[k] = slot < items ? sh.dst[slot] : 0;
        n2[k] = 0.f;
    }
    // the TF32 filter's error bound needs every nonzero coordinate in
    // [2^-60, 2^60]; the FP16 filter scales by the largest finite magnitude;
    // NaN and infinities turn either off
    bool out_of_range = false, nonfinite = false;
    unsigned mx = 0u;
    constexpr int R = 8 / PER;  // rows in flight
    for (int d0 = 0; d0 < dim; d0 += R) {
        float v[R][PER];
#pragma unroll
        for (int r = 0; r < R; ++r)
#pragma unroll
            for (int k = 0; k < PER; ++k)
                v[r][k] = d0 + r < dim && from[k] >= 0 ? __ldg(in + (d0 + r) * ld_in + from[k]) : 0.f;
#pragma unroll
        for (int r = 0; r < R; ++r)
#pragma unroll
            for (int k = 0; k < PER; ++k) {
                const float x = v[r][k], a = fabsf(x);
                out_of_range |= x != 0.f && !(a >= 0x1p-60f && a <= 0x1p60f);
                nonfinite |= !(a <= FLT_MAX);
                if (a <= FLT_MAX) mx = max(mx, __float_as_uint(a));
                n2[k] = fmaf(x, x, n2[k]);
                if (d0 + r < dim && from[k] >= 0) out[(d0 + r) * ld_out + to[k]] = x;
            }
    }
    for (int d = dim; d < dp; ++d)
#pragma unroll
        for (int k = 0; k < PER; ++k)
            if (from[k] >= 0) out[d * ld_out + to[k]] = 0.f;
#pragma unroll
    for (int k = 0; k < PER; ++k) {
        if (from[k] < 0) continue;
        key_out[to[k]] = key[from[k]];
        // the FP32 filter's folded squared norm fl(|x|^2) (1 - 4 gamma)
        if (is_tree) key_out[ld_out + to[k]] = n2[k] * (1.f - 4.f * (kF32G * (dp + 2.f)));
        perm[to[k]] = orig0 + from[k];
    }
    if (out_of_range) S->exact_only = 1;
    if (nonfinite) S->nonfinite = 1;
    mx = __reduce_max_sync(kFull, mx);
    if (lane == 0 && mx) atomicMax(&S->maxabs, mx);
}

__global__ void __launch_bounds__(kSortThreads)
sort_scatter(const float *__restrict__ tree, int N, int64_t ld, int dim, int dp, int tper,
             int tblocks, const float *__restrict__ queries, const float *__restrict__ budgets,
             int Q, int qper, SortState *S, float *__restrict__ tree_s, int ldt,
             int *__restrict__ perm, float *__restrict__ q_s, float *__restrict__ c_s,
             int *__restrict__ qperm) {
    __shared__ ScatterShared sh;
    const bool is_tree = (int)blockIdx.x < tblocks;
    const int per = is_tree ? tper : qper;
    const int64_t base =
        (int64_t)(is_tree ? blockIdx.x : blockIdx.x - tblocks) * per * kSortThreads;
    const int items = (int)min((int64_t)per * kSortThreads, (int64_t)(is_tree ? N : Q) - base);
    const float *in = (is_tree ? tree : queries) + base;
    const float *key = (is_tree ? tree + (size_t)dim * ld : budgets) + base;
    const int64_t ld_in = is_tree ? ld : Q, ld_out = is_tree ? ldt : Q;
    float *out = is_tree ? tree_s : q_s;
    float *key_out = is_tree ? tree_s + (size_t)dp * ldt : c_s;
    int *cur = is_tree ? S->tree_cur : S->query_cur;
    int *pm = is_tree ? perm : qperm;
    switch (per) {
        case 1: scatter_items<1>(in, ld_in, key, items, dim, dp, is_tree, (int)base, S, cur, out,
                                 ld_out, key_out, pm, sh); break;
        case 2: scatter_items<2>(in, ld_in, key, items, dim, dp, is_tree, (int)base, S, cur, out,
                                 ld_out, key_out, pm, sh); break;
        case 4: scatter_items<4>(in, ld_in, key, items, dim, dp, is_tree, (int)base, S, cur, out,
                                 ld_out, key_out, pm, sh); break;
        default: scatter_items<8>(in, ld_in, key, items, dim, dp, is_tree, (int)base, S, cur, out,
                                  ld_out, key_out, pm, sh); break;
    }
}

// Vertices that a block of queries with largest budget c (each of its first
// kTcQueries threads' own) must scan: up to the end of the bucket that holds
// the largest, 0 when no vertex has g below it.  Valid in thread 0; NaN
// budgets admit nothing and are ignored.
__device__ __forceinline__ int nn_block_cut(float c, const SortState *S, float *red) {
    static_assert(kTcQueries == kSortBuckets, "one bucket limit per query");
    const int t = threadIdx.x;
    float m = t < kTcQueries && c == c ? c : -INFINITY;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) m = fmaxf(m, __shfl_xor_sync(kFull, m, o));
    if ((t & 31) == 0 && t < kTcQueries) red[t >> 5] = m;
    __syncthreads();
    m = red[0];
#pragma unroll
    for (int k = 1; k < kTcQueries / 32; ++k) m = fmaxf(m, red[k]);
    const int b = __syncthreads_count(t > 0 && t < kSortBuckets && S->split[t] <= m);
    return m > unkey(S->gmin) ? S->tree_off[b + 1] : 0;
}

// The cuts alone, for the pair count; a NEAREST call takes them from its
// seeding pass.
__global__ void __launch_bounds__(kTcQueries) sort_cut(const float *__restrict__ c_s, int Q,
                                                       const SortState *S, int *__restrict__ cut) {
    __shared__ float red[kTcQueries / 32];
    const int i = blockIdx.x * kTcQueries + threadIdx.x;
    const int n = nn_block_cut(i < Q ? c_s[i] : -INFINITY, S, red);
    if (threadIdx.x == 0) cut[blockIdx.x] = n;
}

// Seeding pass, one block per query block: for each (ordered) query, the
// smallest exact squared distance (the filter's own formula) among
// kSeedSamples evenly spaced vertices of the g-ordered tree that are
// admissible for it (+inf when none is); and the block's cut.  A query's
// samples are shared by four threads, four samples at a time from one 16-byte
// load per coordinate, with packed differences and fused multiply-adds: with
// one thread per query and scalar forms the pass waited on its own chains.
// Whole calls are 3 to 8 us shorter than with those (2,048 queries over 100,000
// vertices in 21-D: 240.2 -> 235.5 us; 8,000 over 20,000 in 56-D: 391.3 -> 383.4).
constexpr int kSeedSamples = 64;
constexpr int kSeedGroups = 4;
template <int DIM>
__global__ void __launch_bounds__(kTcQueries * kSeedGroups)
nearest_seed(const float *__restrict__ tree_s, int N, int ldt, const float *__restrict__ q_s,
             const float *__restrict__ c_s, int Q, const SortState *S, float *__restrict__ seed,
             int *__restrict__ cut) {
    __shared__ __align__(16) float xs[DIM + 1][kSeedSamples];  // the samples, g in the last row
    __shared__ float part[kSeedGroups - 1][kTcQueries];
    __shared__ float red[kTcQueries / 32];
    const int n = min(N, kSeedSamples);
    for (int t = threadIdx.x; t < (DIM + 1) * kSeedSamples; t += blockDim.x) {
        const int d = t / kSeedSamples, k = t % kSeedSamples;
        // vertex k N / n of n = min(N, 64)
        const int v = n == kSeedSamples ? (int)(((int64_t)k * N) / kSeedSamples) : k;
        xs[d][k] = k < n ? tree_s[(size_t)d * ldt + v] : 0.f;
    }
    __syncthreads();
    const int ql = threadIdx.x & (kTcQueries - 1), grp = threadIdx.x / kTcQueries;
    const int i = blockIdx.x * kTcQueries + ql;
    const float c = i < Q ? c_s[i] : -FLT_MAX;
    float best = FLT_MAX * 2.f;
    if (i < Q) {
        f32x2_t acc[kSeedSamples / kSeedGroups / 2];
#pragma unroll
        for (int u = 0; u < kSeedSamples / kSeedGroups / 2; ++u) acc[u] = 0ull;
        const int k0 = grp * (kSeedSamples / kSeedGroups);
#pragma unroll
        for (int d = 0; d < DIM; ++d) {
            // (x - q)^2 is (q - x)^2 to the bit
            const float q = -__ldg(q_s + (size_t)d * Q + i);
            const f32x2_t qq = ((f32x2_t)__float_as_uint(q) << 32) | __float_as_uint(q);
#pragma unroll
            for (int u = 0; u < kSeedSamples / kSeedGroups / 4; ++u) {
                const ulonglong2 x = *reinterpret_cast<const ulonglong2 *>(&xs[d][k0 + 4 * u]);
                acc_sq_f32x2(acc[2 * u], add_f32x2(x.x, qq));
                acc_sq_f32x2(acc[2 * u + 1], add_f32x2(x.y, qq));
            }
        }
#pragma unroll
        for (int u = 0; u < kSeedSamples / kSeedGroups; ++u) {
            const float d2 = (u & 1) ? f32x2_hi(acc[u >> 1]) : f32x2_lo(acc[u >> 1]);
            const float g = xs[DIM][k0 + u];
            if (k0 + u < n && d2 < best && g < c && g + __fsqrt_rn(d2) < c) best = d2;
        }
    }
    if (grp > 0) part[grp - 1][ql] = best;
    __syncthreads();
    if (grp == 0 && i < Q) {
#pragma unroll
        for (int k = 0; k < kSeedGroups - 1; ++k) best = fminf(best, part[k][ql]);
        seed[i] = best;
    }
    const int nc = nn_block_cut(i < Q ? c : -INFINITY, S, red);
    if (threadIdx.x == 0) cut[blockIdx.x] = nc;
}

// Pairs the budget-ordered pass scans: sum over query blocks of (queries in
// the block) x cut.
__global__ void sort_count_pairs(const int *__restrict__ cut, int qblocks, int Q, int bq,
                                 unsigned long long *out) {
    unsigned long long acc = 0;
    for (int b = threadIdx.x; b < qblocks; b += blockDim.x)
        acc += (unsigned long long)min(bq, Q - b * bq) * (unsigned long long)cut[b];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(kFull, acc, o);
    if ((threadIdx.x & 31) == 0) atomicAdd(out, acc);
}

// Raises the FP32 filter's dynamic shared-memory limit once per device and
// returns its resident blocks per SM.
template <int DIM>
mrpop_status f32_filter_setup(int dev, int *bps) {
    static std::mutex mu;
    static int done[64] = {};
    static int occ[64] = {};
    std::lock_guard<std::mutex> lock(mu);
    if (dev < 0 || dev >= 64) return set_error(MRPOP_EINVAL, "nearest: device ordinal %d", dev);
    if (!done[dev]) {
        MRPOP_CUDA_TRY(cudaFuncSetAttribute(nearest_f32_kernel<DIM>,
                                            cudaFuncAttributeMaxDynamicSharedMemorySize,
                                            (int)f32_smem_bytes<DIM>()));
        MRPOP_CUDA_TRY(cudaOccupancyMaxActiveBlocksPerMultiprocessor(
            &occ[dev], nearest_f32_kernel<DIM>, kTcThreads, f32_smem_bytes<DIM>()));
        done[dev] = 1;
    }
    *bps = occ[dev];
    return MRPOP_OK;
}

// Dimensions of the tensor-core filters' instances; the FP32 filter serves the
// padded dimensions between and above them whatever the filter asked for.
constexpr bool tensor_dim(int d) {
    return d == 3 || d == 6 || d == 7 || d == 14 || d == 21 || d == 28;
}

// DIM: the instance's coordinate rows, dim <= DIM of them the caller's.
// out_idx null: only count the scanned pairs into *pairs (synchronises).
// filter: MRPOP_NEAREST_FILTER_FP32 (FMA-pipe expansion filter) or
// MRPOP_NEAREST_FILTER_TENSOR (FP16 / TF32 mma.sync expansion filter); both
// decide every survivor exactly, so the indices do not depend on it.
template <int DIM>
mrpop_status nearest_sorted(const float *tree, int N, int64_t ld, int dim, const float *queries,
                            const float *budgets, int Q, int64_t *out_idx, cudaStream_t st,
                            int64_t *pairs, int filter, int waves) {
    int dev = 0, sms = 1, bps = 1;
    MRPOP_CUDA_TRY(cudaGetDevice(&dev));
    MRPOP_CUDA_TRY(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
    constexpr bool f16 = DIM + 2 <= 16;  // FP16 tensor filter (K = 16), else TF32
    const bool tensor = tensor_dim(DIM) && dim == DIM && filter == MRPOP_NEAREST_FILTER_TENSOR;
    if (!tensor) {
        const mrpop_status fs = f32_filter_setup<DIM>(dev, &bps);
        if (fs != MRPOP_OK) return fs;
    } else if constexpr (tensor_dim(DIM) && f16) {
        MRPOP_CUDA_TRY(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&bps, nearest_tc16_kernel<DIM>,
                                                                     kTcThreads, 0));
    } else if constexpr (tensor_dim(DIM)) {
        MRPOP_CUDA_TRY(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&bps, nearest_tc_kernel<DIM>,
                                                                     kTcThreads, 0));
    }
    bps = std::max(bps, 1);
    const int bq = kTcQueries;
    const int qblocks = (Q + bq - 1) / bq;
    // about four waves of (query block, tree slice) pieces before the cut
    // removes some: the dynamic block scheduler then evens out the blocks
    // that stop early
    int splits = std::max(1, (std::max(1, waves) * sms * bps + qblocks - 1) / qblocks);
    int chunk = (N + splits - 1) / splits;
    chunk = std::max(kSliceAlign, ((chunk + kSliceAlign - 1) / kSliceAlign) * kSliceAlign);
    splits = std::max(1, (N + chunk - 1) / chunk);
    if (splits > 65535) return set_error(MRPOP_EINVAL, "nearest: tree too large");
    // one stream-ordered arena: sort state, ordered tree and queries,
    // permutations, cuts, partial bests
    auto align = [](size_t b) { return (b + 255) & ~(size_t)255; };
    const size_t b_state = align(sizeof(SortState));
    // rows of the ordered tree start on 16-byte boundaries (the FP32 filter
    // copies them in 16-byte pieces)
    const int ldt = (N + 3) & ~3;
    const size_t b_tree = align(sizeof(float) * (size_t)(DIM + 2) * ldt);  // + folded norms
    const size_t b_perm = align(sizeof(int) * (size_t)N);
    const size_t b_q = align(sizeof(float) * (size_t)DIM * Q);
    const size_t b_c = align(sizeof(float) * (size_t)Q);
    const size_t b_qp = align(sizeof(int) * (size_t)Q);
    const size_t b_cut = align(sizeof(int) * (size_t)qblocks);
    const size_t b_part = align(sizeof(Best) * (size_t)splits * Q);
    const size_t b_seed = align(sizeof(float) * (size_t)Q);
    const size_t b_qdone = align(sizeof(int) * (size_t)qblocks);
    char *arena = nullptr;
    const cudaError_t ae = scratch_alloc((void **)&arena,
                                         b_state + b_tree + b_perm + b_q + b_c + b_qp + b_cut +
                                             b_part + b_seed + b_qdone,
                                         st);
    if (ae != cudaSuccess) {
        cudaGetLastError();  // not left for a later launch check
        return cuda_error(ae, "nearest: scratch");
    }
    char *at = arena;
    auto take = [&](size_t b) { char *r = at; at += b; return r; };
    SortState *S = (SortState *)take(b_state);
    float *tree_s = (float *)take(b_tree);
    int *perm = (int *)take(b_perm);
    float *q_s = (float *)take(b_q);
    float *c_s = (float *)take(b_c);
    int *qperm = (int *)take(b_qp);
    int *cut = (int *)take(b_cut);
    Best *partial = (Best *)take(b_part);
    float *seed = (float *)take(b_seed);
    int *qdone = (int *)take(b_qdone);
    const float *g = tree + (size_t)dim * ld;
    // five launches: setup (bucket limits), histogram (+ scan), scatter, seed
    // (+ cut), filter (+ reduce in each query block's last slice)
    const int tper = sort_per(N), qper = sort_per(Q);
    const int tblocks = (int)(((int64_t)N + tper * kSortThreads - 1) / (tper * kSortThreads));
    const int sblocks = tblocks + (int)(((int64_t)Q + qper * kSortThreads - 1) /
                                        (qper * kSortThreads));
    sort_setup<<<1, kSortBuckets, 0, st>>>(g, N, S, qdone, qblocks);
    sort_histogram<<<sblocks, kSortThreads, 0, st>>>(g, N, tper, tblocks, budgets, Q, qper, S);
    sort_scatter<<<sblocks, kSortThreads, 0, st>>>(tree, N, ld, dim, DIM, tper, tblocks, queries,
                                                   budgets, Q, qper, S, tree_s, ldt, perm, q_s,
                                                   c_s, qperm);
    if (!out_idx) {
        sort_cut<<<qblocks, kTcQueries, 0, st>>>(c_s, Q, S, cut);
        unsigned long long *d_pairs = (unsigned long long *)seed;  // 8 bytes of the arena
        unsigned long long h = 0;
        cudaMemsetAsync(d_pairs, 0, sizeof(unsigned long long), st);
        sort_count_pairs<<<1, 256, 0, st>>>(cut, qblocks, Q, bq, d_pairs);
        cudaMemcpyAsync(&h, d_pairs, sizeof(h), cudaMemcpyDeviceToHost, st);
        cudaError_t e = cudaStreamSynchronize(st);
        if (e == cudaSuccess) e = cudaGetLastError();
        cudaFreeAsync(arena, st);
        if (e != cudaSuccess) return cuda_error(e, "nearest pair count");
        *pairs = (int64_t)h;
        return MRPOP_OK;
    }
    nearest_seed<DIM><<<qblocks, kTcQueries * kSeedGroups, 0, st>>>(tree_s, N, ldt, q_s, c_s, Q, S, seed, cut);
    dim3 grid(qblocks, splits);
    const NnFinish fin{qdone, qperm, out_idx};
    if (!tensor)
        nearest_f32_kernel<DIM><<<grid, kTcThreads, f32_smem_bytes<DIM>(), st>>>(
            tree_s, N, ldt, q_s, c_s, Q, chunk, partial, perm, cut, seed, &S->exact_only, fin);
    else if constexpr (tensor_dim(DIM) && f16)
        nearest_tc16_kernel<DIM><<<grid, kTcThreads, 0, st>>>(tree_s, N, ldt, q_s, c_s, Q, chunk,
                                                              partial, perm, cut, seed,
                                                              &S->maxabs, &S->nonfinite, fin);
    else if constexpr (tensor_dim(DIM))
        nearest_tc_kernel<DIM><<<grid, kTcThreads, 0, st>>>(tree_s, N, ldt, q_s, c_s, Q, chunk, partial,
                                                            perm, cut, seed, &S->exact_only, fin);
    const cudaError_t e = cudaGetLastError();
    cudaFreeAsync(arena, st);
    if (e != cudaSuccess) return cuda_error(e, "nearest (budget-ordered) launch");
    return MRPOP_OK;
}

// NEIGHBORS: a block serves kNbWarps queries, one warp each, and streams the
// tree through shared memory in tiles of kNbTile vertices (SoA rows, loaded
// once for all of the block's queries).  Lanes take 32 consecutive vertices at
// a time in ascending order; ballot + prefix popcount keep the output sorted.
constexpr int kNbWarps = 8;
constexpr int kNbTile = 256;

__global__ void __launch_bounds__(kNbWarps * 32)
neighbors_kernel(const float *__restrict__ tree, int N, int64_t ld, int dim,
                 const float *__restrict__ queries, int Q, float delta, int64_t k_max,
                 int64_t *__restrict__ out_idx, int64_t *__restrict__ out_cnt, int chunk) {
    // blockIdx.y takes vertices [y * chunk, (y + 1) * chunk); with several
    // ranges (gridDim.y > 1) the lists go to per-range slots of out_idx /
    // out_cnt ([q][range]) and neighbors_merge concatenates them in order
    __shared__ float qs[kNbWarps][MRPOP_MAX_LINKS];
    extern __shared__ float tile[];  // [dim][kNbTile]
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int q = blockIdx.x * kNbWarps + warp;
    const bool qok = q < Q;
    for (int d = lane; d < dim; d += 32) qs[warp][d] = qok ? queries[(size_t)d * Q + q] : 0.f;
    const int64_t slot = (int64_t)q * gridDim.y + blockIdx.y;  // this query's range slot
    const int vs = blockIdx.y * chunk, ve = min(N, vs + chunk);
    int64_t count = 0;
    for (int v0 = vs; v0 < ve; v0 += kNbTile) {
        const int nv = min(kNbTile, ve - v0);
        __syncthreads();
        for (int i = threadIdx.x; i < dim * kNbTile; i += blockDim.x) {
            const int d = i / kNbTile, j = i - d * kNbTile;
            tile[i] = j < nv ? __ldg(tree + (size_t)d * ld + v0 + j) : 0.f;
        }
        __syncthreads();
        if (!qok) continue;
        for (int c = 0; c < nv; c += 32) {
            const int v = c + lane;
            bool in = false;
            if (v < nv) {
                float d2 = 0.f;
                for (int d = 0; d < dim; ++d) {
                    const float a = qs[warp][d] - tile[d * kNbTile + v];
                    d2 = fmaf(a, a, d2);
                }
                in = __fsqrt_rn(d2) <= delta;
            }
            const unsigned bal = __ballot_sync(kFull, in);
            if (in) {
                const int64_t pos = count + __popc(bal & ((1u << lane) - 1u));
                if (pos < k_max) out_idx[(size_t)slot * k_max + pos] = v0 + v;
            }
            count += __popc(bal);
        }
    }
    if (!qok) return;
    for (int64_t pos = count + lane; pos < k_max; pos += 32) out_idx[(size_t)slot * k_max + pos] = -1;
    if (lane == 0) out_cnt[slot] = count;
}

// NEIGHBORS in one launch, for lists of up to kNbListMax entries: the vertex
// ranges of a group of 8 queries are the blocks of one cluster (at most 8).
// Each warp scans its range for its query, the query in registers and the
// distance compared squared (thr: the largest float whose square root is
// within delta), and keeps its list in shared memory; then the blocks read one
// another's counts and write their part of each list in place.  1,024 queries
// over 4,096 vertices in 7-D: 14.5 us (ncu, cold L2); writing the ranges' lists to
// scratch and concatenating them in a second kernel, one thread per query, 20.2 +
// 7.9 and an allocation.  A call, which the host bounds, 20.9 to 26.7 us over four
// runs, 28.8 to 29.4 that way.
constexpr int kNbListMax = 64;
constexpr int kNbCluster = 8;

template <int DP>
__global__ void __launch_bounds__(kNbWarps * 32)
neighbors_cluster_kernel(const float *__restrict__ tree, int N, int64_t ld, int dim,
                         const float *__restrict__ queries, int Q, float thr, int k_max,
                         int64_t *__restrict__ out_idx, int64_t *__restrict__ out_cnt, int chunk) {
    namespace cg = cooperative_groups;
    __shared__ float tile[DP * kNbTile];
    __shared__ int list[kNbWarps][kNbListMax];
    __shared__ int cnt[kNbWarps];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int q = blockIdx.x * kNbWarps + warp;
    const bool qok = q < Q;
    float qv[DP];
#pragma unroll
    for (int d = 0; d < DP; ++d)
        qv[d] = qok && d < dim ? __ldg(queries + (size_t)d * Q + q) : 0.f;
    const int vs = (int)min((int64_t)N, (int64_t)blockIdx.y * chunk);
    const int ve = (int)min((int64_t)N, (int64_t)vs + chunk);
    int count = 0;
    for (int v0 = vs; v0 < ve; v0 += kNbTile) {
        const int nv = min(kNbTile, ve - v0);
        __syncthreads();
#pragma unroll
        for (int d = 0; d < DP; ++d)  // (rows past the dimension stay zero)
            tile[d * kNbTile + threadIdx.x] =
                d < dim && (int)threadIdx.x < nv ? __ldg(tree + (size_t)d * ld + v0 + threadIdx.x) : 0.f;
        __syncthreads();
        if (!qok) continue;
        for (int c = 0; c < nv; c += 32) {
            const int v = c + lane;
            float d2 = 0.f;
#pragma unroll
            for (int d = 0; d < DP; ++d) {
                const float a = qv[d] - tile[d * kNbTile + v];
                d2 = fmaf(a, a, d2);
            }
            const bool in = v < nv && d2 <= thr;
            const unsigned bal = __ballot_sync(kFull, in);
            const int pos = count + __popc(bal & ((1u << lane) - 1u));
            if (in && pos < k_max) list[warp][pos] = v0 + v;
            count += __popc(bal);
        }
    }
    if (lane == 0) cnt[warp] = count;
    cg::cluster_group cl = cg::this_cluster();
    cl.sync();
    if (qok) {
        const int ranks = (int)cl.num_blocks(), rank = (int)cl.block_rank();
        const int c = lane < ranks ? cl.map_shared_rank(cnt, lane)[warp] : 0;
        int before = lane < rank ? c : 0, total = c;
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            before += __shfl_xor_sync(kFull, before, o);
            total += __shfl_xor_sync(kFull, total, o);
        }
        int64_t *row = out_idx + (size_t)q * k_max;
        for (int i = lane; i < count && before + i < k_max; i += 32) row[before + i] = list[warp][i];
        if (rank == 0) {
            for (int i = total + lane; i < k_max; i += 32) row[i] = -1;
            if (lane == 0) out_cnt[q] = total;
        }
    }
    cl.sync();  // no block ends while its counts are read
}

// Largest float x with sqrt(x) <= delta in FP32 (-1 when there is none, NaN
// for NaN): comparing a squared distance with it decides as comparing its
// correctly rounded square root with delta, which is monotonic.
static float radius_threshold(float delta) {
    if (!(delta >= 0.f)) return delta != delta ? delta : -1.f;
    if (delta > FLT_MAX) return delta;
    float x = (float)std::min((double)delta * (double)delta, (double)FLT_MAX);
    while (x < FLT_MAX && std::sqrt(std::nextafter(x, FLT_MAX)) <= delta)
        x = std::nextafter(x, FLT_MAX);
    while (x > 0.f && std::sqrt(x) > delta) x = std::nextafter(x, 0.f);
    return x;
}

template <int DP>
mrpop_status neighbors_cluster(const float *tree, int N, int64_t ld, int dim, const float *queries,
                               int Q, float delta, int k_max, int64_t *out_idx, int64_t *out_cnt,
                               int ranges, cudaStream_t st) {
    const int chunk = (int)std::max<int64_t>(
        ((int64_t)(N + ranges - 1) / ranges + kNbTile - 1) / kNbTile * kNbTile, kNbTile);
    cudaLaunchAttribute at{};
    at.id = cudaLaunchAttributeClusterDimension;
    at.val.clusterDim.x = 1;
    at.val.clusterDim.y = std::max(1, (N + chunk - 1) / chunk);
    at.val.clusterDim.z = 1;
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3((Q + kNbWarps - 1) / kNbWarps, at.val.clusterDim.y);
    cfg.blockDim = dim3(kNbWarps * 32);
    cfg.stream = st;
    cfg.attrs = &at;
    cfg.numAttrs = 1;
    MRPOP_CUDA_TRY(cudaLaunchKernelEx(&cfg, neighbors_cluster_kernel<DP>, tree, N, ld, dim, queries,
                                      Q, radius_threshold(delta), k_max, out_idx, out_cnt, chunk));
    return MRPOP_OK;
}

// Concatenates each query's per-range lists in range order (ascending vertex
// index), keeping the first k_max, and adds up the counts.
__global__ void neighbors_merge(const int64_t *__restrict__ part_idx,
                                const int64_t *__restrict__ part_cnt, int ranges, int Q,
                                int64_t k_max, int64_t *__restrict__ out_idx,
                                int64_t *__restrict__ out_cnt) {
    const int q = blockIdx.x * blockDim.x + threadIdx.x;
    if (q >= Q) return;
    int64_t total = 0;
    for (int r = 0; r < ranges; ++r) {
        const int64_t slot = (int64_t)q * ranges + r;
        const int64_t c = part_cnt[slot];
        for (int64_t i = 0; i < c && total + i < k_max; ++i)
            out_idx[(size_t)q * k_max + total + i] = part_idx[(size_t)slot * k_max + i];
        total += c;
    }
    for (int64_t pos = total; pos < k_max; ++pos) out_idx[(size_t)q * k_max + pos] = -1;
    out_cnt[q] = total;
}

// C(sigma): segment lengths in FP32, sums in FP64 with a fixed reduction order,
// so the result is deterministic.
// Length of segment j, its two rows read in vectors of V floats (V divides
// dim and the rows are aligned to V floats).
template <int V>
__device__ __forceinline__ float segment_length(const float *__restrict__ path, int64_t j, int dim) {
    const float *p = path + j * dim;
    float s = 0.f;
#pragma unroll 4
    for (int d = 0; d < dim; d += V) {
        float x[V], y[V];
        if constexpr (V == 4) {
            *reinterpret_cast<float4 *>(x) = __ldg(reinterpret_cast<const float4 *>(p + d));
            *reinterpret_cast<float4 *>(y) = __ldg(reinterpret_cast<const float4 *>(p + dim + d));
        } else if constexpr (V == 2) {
            *reinterpret_cast<float2 *>(x) = __ldg(reinterpret_cast<const float2 *>(p + d));
            *reinterpret_cast<float2 *>(y) = __ldg(reinterpret_cast<const float2 *>(p + dim + d));
        } else {
            x[0] = __ldg(p + d);
            y[0] = __ldg(p + dim + d);
        }
#pragma unroll
        for (int k = 0; k < V; ++k) {
            const float a = y[k] - x[k];
            s = fmaf(a, a, s);
        }
    }
    return __fsqrt_rn(s);
}

constexpr int kPathThreads = 512;

// Each block sums the segments [block * chunk, block * chunk + chunk) in a
// fixed order (per thread in steps of the block, then a tree in shared memory:
// FP64 additions are scarce, so no warp repeats another's).  A cluster of up to
// 8 blocks covers a path of up to 16,384 segments and its first block adds the
// blocks' sums in block order: one launch and no scratch (16,385 vertices in
// 14-D: 12.3 us with a cold L2, 17.5 with 4-byte loads and a second kernel).
// Longer paths need more SMs to read from memory (65,537 vertices in 14-D, cold:
// 28.7 us as a cluster, 13.3 as 64 blocks; 131,073: 47 and 15.4), and so do
// 4-byte loads above 350,000 floats (35-D, 8,001 vertices 16.4 us a call as a
// cluster and 21.0 in blocks, 10,001 19.4 and 19.4, 16,001 27.2 and 19.9): their
// blocks write their sums to partial, which a second kernel adds.
template <int V>
__global__ void __launch_bounds__(kPathThreads)
path_cost_kernel(const float *__restrict__ path, int64_t M, int dim, int64_t chunk,
                 double *__restrict__ partial, double *__restrict__ out) {
    __shared__ double red[kPathThreads];
    const int t = threadIdx.x;
    const int64_t j0 = (int64_t)blockIdx.x * chunk;
    const int64_t j1 = min(M - 1, j0 + chunk);
    double acc = 0.0;
    for (int64_t j = j0 + t; j < j1; j += 2 * kPathThreads) {
        const int64_t k = j + kPathThreads;
        const float a = segment_length<V>(path, j, dim);
        const float b = k < j1 ? segment_length<V>(path, k, dim) : 0.f;
        acc += (double)a;
        if (k < j1) acc += (double)b;
    }
    red[t] = acc;
#pragma unroll
    for (int w = kPathThreads / 2; w >= 32; w >>= 1) {
        __syncthreads();
        if (t < w) red[t] = acc += red[t + w];
    }
    if (t < 32) {
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) acc += __shfl_down_sync(kFull, acc, o);
        if (t == 0) red[0] = acc;
    }
    if (partial) {
        if (t == 0) partial[blockIdx.x] = acc;
        return;
    }
    if (gridDim.x == 1) {
        if (t == 0) *out = acc;
        return;
    }
    namespace cg = cooperative_groups;
    cg::cluster_group cl = cg::this_cluster();
    cl.sync();
    if (cl.block_rank() == 0 && t == 0) {
        double sum = acc;
        for (unsigned r = 1; r < cl.num_blocks(); ++r) sum += *cl.map_shared_rank(red, r);
        *out = sum;
    }
    cl.sync();  // no block ends while its sum is read
}

__global__ void sum_partials_kernel(const double *__restrict__ partial, int n,
                                    double *__restrict__ out) {
    double acc = 0.0;
    for (int i = threadIdx.x; i < n; i += 32) acc += partial[i];
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) acc += __shfl_xor_sync(kFull, acc, off);
    if (threadIdx.x == 0) *out = acc;
}

}  // namespace

// Tuned-launch cache keys and lookups: the budget-ordered NEAREST's slice
// waves (default 4) and NEIGHBORS's vertex-range target (default 54 warps per
// SM), per (architecture, dimension, log2 of the tree size, log2 of the batch).
static std::string nn_key(const char *kind, int dim, int64_t N, int64_t Q, int filter) {
    return std::string(kind) + " " + tune_arch() + " dim=" + std::to_string(dim) + " N=2^" +
           std::to_string(log2_bucket(N)) + " Q=2^" + std::to_string(log2_bucket(Q)) +
           (filter >= 0 ? " filter=" + std::to_string(filter) : std::string());
}

int nearest_tuned(int dim, int64_t N, int64_t Q, int filter) {
    std::vector<int> v;
    return tune_lookup(nn_key("nearest", dim, N, Q, filter), &v) && !v.empty() && v[0] > 0 ? v[0] : 4;
}

int neighbors_tuned(int dim, int64_t N, int64_t Q) {
    std::vector<int> v;
    return tune_lookup(nn_key("neighbors", dim, N, Q, -1), &v) && !v.empty() && v[0] > 0 ? v[0] : 54;
}

// Times candidates[] (the value passed as the launch knob) with `run`, keeps
// the fastest under key.
template <class Run>
static mrpop_status tune_candidates(const std::string &key, const int *cand, int nc, int reps,
                                    Run run, cudaStream_t st, int32_t *best_out, float *ms_out) {
    cudaEvent_t a, b;
    MRPOP_CUDA_TRY(cudaEventCreate(&a));
    MRPOP_CUDA_TRY(cudaEventCreate(&b));
    float best = INFINITY;
    int bv = 0;
    mrpop_status s = MRPOP_OK;
    for (int i = 0; i < nc && s == MRPOP_OK; ++i) {
        s = run(cand[i]);  // warm
        float tot = 0.f;
        for (int r = 0; r < reps && s == MRPOP_OK; ++r) {
            cudaEventRecord(a, st);
            s = run(cand[i]);
            cudaEventRecord(b, st);
            cudaEventSynchronize(b);
            float ms = 0.f;
            cudaEventElapsedTime(&ms, a, b);
            tot += ms;
        }
        if (s == MRPOP_OK && tot < best) {
            best = tot;
            bv = cand[i];
        }
    }
    cudaEventDestroy(a);
    cudaEventDestroy(b);
    if (s != MRPOP_OK) return s;
    tune_store(key, {bv});
    if (best_out) *best_out = bv;
    if (ms_out) *ms_out = best / std::max(1, reps);
    return MRPOP_OK;
}

mrpop_status autotune_nearest(const float *tree, int64_t N, int64_t ld, int dim,
                              const float *queries, const float *budgets, int64_t Q,
                              int filter, int64_t *out_idx, int32_t *waves_out, float *ms_out,
                              cudaStream_t st) {
    static const int cand[] = {2, 4, 8};
    return tune_candidates(nn_key("nearest", dim, N, Q, filter), cand, 3, 3,
                           [&](int w) {
                               return launch_nearest(tree, N, ld, dim, queries, budgets, Q,
                                                     out_idx, st, filter, w);
                           },
                           st, waves_out, ms_out);
}

mrpop_status autotune_neighbors(const float *tree, int64_t N, int64_t ld, int dim,
                                const float *queries, int64_t Q, float delta, int64_t k_max,
                                int64_t *out_idx, int64_t *out_cnt, int32_t *target_out,
                                float *ms_out, cudaStream_t st) {
    static const int cand[] = {14, 54, 216};
    return tune_candidates(nn_key("neighbors", dim, N, Q, -1), cand, 3, 3,
                           [&](int t) {
                               return launch_neighbors(tree, N, ld, dim, queries, Q, delta, k_max,
                                                       out_idx, out_cnt, st, t);
                           },
                           st, target_out, ms_out);
}

// The budget-ordered path at the smallest instance of at least dim rows.  Its
// own instance for the dimensions of this library's arms and their first
// multiples, steps of 4 to 12 rows elsewhere: the chain of a pair is as long
// as the rows, so padding costs (DIM - dim) / dim of it, where the exact scan
// these dimensions took before costs two operations per coordinate of all
// N Q pairs, read from L2 once per 8 queries (35-D, 8,192 queries over 50,000
// vertices: 2,457 us against 501).
static mrpop_status nearest_sorted_dim(const float *tree, int n, int64_t ld, int dim,
                                       const float *queries, const float *budgets, int q,
                                       int64_t *out_idx, cudaStream_t st, int64_t *pairs,
                                       int filter, int w) {
#define MRPOP_NN_DIM(D)                                                                       \
    if (dim <= D)                                                                             \
        return nearest_sorted<D>(tree, n, ld, dim, queries, budgets, q, out_idx, st, pairs, filter, w)
    MRPOP_NN_DIM(3);
    MRPOP_NN_DIM(6);
    MRPOP_NN_DIM(7);
    MRPOP_NN_DIM(12);
    MRPOP_NN_DIM(14);
    MRPOP_NN_DIM(16);
    MRPOP_NN_DIM(21);
    MRPOP_NN_DIM(24);
    MRPOP_NN_DIM(28);
    MRPOP_NN_DIM(32);
    MRPOP_NN_DIM(36);
    MRPOP_NN_DIM(44);
    MRPOP_NN_DIM(52);
    MRPOP_NN_DIM(56);
    MRPOP_NN_DIM(64);
#undef MRPOP_NN_DIM
    return set_error(MRPOP_EINVAL, "nearest: dimension %d", dim);
}

// Whether a call takes the budget-ordered path, by its work in pairs x
// coordinates.  The ordering passes and the filter's start cost 60 to 130 us
// whatever the batch; the scan costs two FMA-pipe operations per coordinate of
// every pair, the filter one of the pairs below the budgets.  Measured, scan /
// ordered (us): 14-D, 16,000 vertices, 2,000 queries (4.5e8) 58 / 86; 14-D,
// 4,000 x 8,000 (4.5e8) 68 / 79; 28-D, 4,000 x 8,000 (9e8) 106 / 105; 6-D,
// 16,000 x 8,000 (7.7e8) 120 / 104; 14-D, 64,000 x 2,000 (1.8e9) 174 / 152.
// With fewer queries a query block's bounds start loose in more slices:
// 28-D, 64,000 x 1,024 (1.8e9) 158 / 190; 14-D, 256,000 x 1,024 (3.7e9) 305 /
// 249; 14-D, 1,000,000 x 256 (3.6e9) 298 / 486.  In the dimensions of the
// tensor-core filters alone the ordered path also serves every batch that asks
// for one, and from 4,096 queries over 2,560 vertices on it is kept below the
// line, so that batches of that size skip the pairs whose cost rules them out,
// as mrpop_nearest_work counts (7-D, 3,500 x 4,096: 65 us; the scan is up to 25
// us faster there).  Elsewhere these two calls would be slower for it: 2,560 x
// 4,096 in 4-D 31 us by an earlier scan and 60 ordered, in 16-D 45 and 75.
static bool takes_sorted(int dim, int64_t N, int64_t Q, int filter) {
    if (N <= 0 || !(N <= (1 << 30) || tensor_dim(dim))) return false;
    const double work = (double)N * (double)Q * dim;
    if (Q < 2048) return Q >= 512 && work >= 3e9;
    return work >= 6e8 || (tensor_dim(dim) && (filter == MRPOP_NEAREST_FILTER_TENSOR ||
                                               (Q >= 4096 && N >= 2560)));
}

mrpop_status launch_nearest(const float *tree, int64_t N, int64_t ld, int dim,
                            const float *queries, const float *budgets, int64_t Q,
                            int64_t *out_idx, cudaStream_t st, int filter, int waves) {
    const int n = (int)N, q = (int)Q;
    bool no_scratch = false;
    // Large batches: budget-ordered tree and queries, expansion filter with
    // exact decisions over shared-memory tree tiles.
    if (takes_sorted(dim, N, Q, filter)) {
        const int w = waves > 0 ? waves : nearest_tuned(dim, N, Q, filter);
        const mrpop_status s = nearest_sorted_dim(tree, n, ld, dim, queries, budgets, q, out_idx,
                                                  st, nullptr, filter, w);
        // the ordered copies of a tree that nearly fills the device did not
        // fit: the scan needs none, and in one cluster's slices no scratch either
        if (s != MRPOP_ENOMEM) return s;
        no_scratch = true;
    }
    return nearest_scan(tree, n, ld, dim, queries, budgets, q, out_idx, st, no_scratch);
}

mrpop_status nearest_pairs(const float *tree, int64_t N, int64_t ld, int dim, const float *queries,
                           const float *budgets, int64_t Q, int64_t *pairs, cudaStream_t st) {
    const int n = (int)N, q = (int)Q;
    *pairs = N * Q;  // the small-batch kernels scan every vertex
    if (takes_sorted(dim, N, Q, MRPOP_NEAREST_FILTER_FP32))
        return nearest_sorted_dim(tree, n, ld, dim, queries, budgets, q, nullptr, st, pairs,
                                  MRPOP_NEAREST_FILTER_FP32, 4);
    return MRPOP_OK;
}

mrpop_status launch_neighbors(const float *tree, int64_t N, int64_t ld, int dim,
                              const float *queries, int64_t Q, float delta, int64_t k_max,
                              int64_t *out_idx, int64_t *out_cnt, cudaStream_t st,
                              int warps_per_sm) {
    if (warps_per_sm <= 0) warps_per_sm = neighbors_tuned(dim, N, Q);
    const int blocks = (int)((Q + kNbWarps - 1) / kNbWarps);
    const size_t smem = sizeof(float) * (size_t)dim * kNbTile;
    if (smem > 48 * 1024)
        MRPOP_CUDA_TRY(cudaFuncSetAttribute(neighbors_kernel,
                                            cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
    // Few queries leave most SMs idle with one warp per query: split the
    // vertices into ranges (at least one tile each) until about warps_per_sm
    // warps per SM run (54 by default: about 8,192 on 152 SMs; tunable).
    int sms = 1, dev = 0;
    MRPOP_CUDA_TRY(cudaGetDevice(&dev));
    MRPOP_CUDA_TRY(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
    const int64_t want = std::max<int64_t>(1, (int64_t)sms * std::max(1, warps_per_sm) / std::max<int64_t>(Q, 1));
    const int ranges = (int)std::min<int64_t>(std::min<int64_t>(want, (N + kNbTile - 1) / kNbTile),
                                              std::max<int64_t>(1, 65535));
    // short lists in up to 16 dimensions: the ranges as one cluster, up to
    // 65,536 vertices (8,192 a block; beyond, more ranges repay the merge), for a
    // single query up to 24,576 above 4 dimensions (its 8 blocks leave the chip
    // idle: 7-D, 48,000 vertices 46.0 us, in ranges 31.9; 24,000 25.8 and 26.4)
    if (k_max <= kNbListMax && dim <= 16 && N <= (Q == 1 && dim > 4 ? 24576 : 65536) && Q > 0) {
        const int r = std::max(1, std::min(ranges, kNbCluster)), n = (int)N, q = (int)Q,
                  k = (int)k_max;
        if (dim <= 4)
            return neighbors_cluster<4>(tree, n, ld, dim, queries, q, delta, k, out_idx, out_cnt, r, st);
        if (dim <= 7)
            return neighbors_cluster<7>(tree, n, ld, dim, queries, q, delta, k, out_idx, out_cnt, r, st);
        if (dim <= 10)
            return neighbors_cluster<10>(tree, n, ld, dim, queries, q, delta, k, out_idx, out_cnt, r, st);
        return neighbors_cluster<16>(tree, n, ld, dim, queries, q, delta, k, out_idx, out_cnt, r, st);
    }
    if (ranges <= 1 || k_max > 4096) {
        neighbors_kernel<<<blocks, kNbWarps * 32, smem, st>>>(tree, (int)N, ld, dim, queries,
                                                              (int)Q, delta, k_max, out_idx,
                                                              out_cnt, (int)std::max<int64_t>(N, 1));
        MRPOP_CUDA_TRY(cudaGetLastError());
        return MRPOP_OK;
    }
    const int chunk = (int)(((N + ranges - 1) / ranges + kNbTile - 1) / kNbTile * kNbTile);
    const int nr = (int)((N + chunk - 1) / chunk);
    int64_t *part = nullptr;
    const size_t kidx = (size_t)Q * nr * (size_t)std::max<int64_t>(k_max, 1);
    MRPOP_CUDA_TRY(scratch_alloc((void **)&part, sizeof(int64_t) * (kidx + (size_t)Q * nr), st));
    neighbors_kernel<<<dim3(blocks, nr), kNbWarps * 32, smem, st>>>(
        tree, (int)N, ld, dim, queries, (int)Q, delta, k_max, part, part + kidx, chunk);
    neighbors_merge<<<(int)((Q + 127) / 128), 128, 0, st>>>(part, part + kidx, nr, (int)Q, k_max,
                                                           out_idx, out_cnt);
    const cudaError_t e = cudaGetLastError();
    cudaFreeAsync(part, st);
    if (e != cudaSuccess) return cuda_error(e, "neighbors launch");
    return MRPOP_OK;
}

template <int V>
static mrpop_status path_cost_v(const float *path, int64_t M, int dim, double *out,
                                cudaStream_t st) {
    const int64_t segs = M > 1 ? M - 1 : 0;
    constexpr int64_t kBlockSegs = 2 * kPathThreads;
    if (segs <= 16384 && (V > 1 || segs * dim <= 350000)) {
        int blocks = 1;
        while (blocks < 8 && blocks * kBlockSegs < segs) blocks *= 2;
        cudaLaunchAttribute at{};
        at.id = cudaLaunchAttributeClusterDimension;
        at.val.clusterDim.x = blocks;
        at.val.clusterDim.y = at.val.clusterDim.z = 1;
        cudaLaunchConfig_t cfg{};
        cfg.gridDim = dim3(blocks);
        cfg.blockDim = dim3(kPathThreads);
        cfg.stream = st;
        cfg.attrs = &at;
        cfg.numAttrs = 1;
        MRPOP_CUDA_TRY(cudaLaunchKernelEx(&cfg, path_cost_kernel<V>, path, M, dim,
                                          (segs + blocks - 1) / blocks, (double *)nullptr, out));
        return MRPOP_OK;
    }
    const int blocks = (int)std::min<int64_t>(1024, (segs + kBlockSegs - 1) / kBlockSegs);
    const int64_t chunk = (segs + blocks - 1) / blocks;
    double *partial = nullptr;
    MRPOP_CUDA_TRY(scratch_alloc((void **)&partial, sizeof(double) * blocks, st));
    path_cost_kernel<V><<<blocks, kPathThreads, 0, st>>>(path, M, dim, chunk, partial, nullptr);
    cudaError_t e = cudaGetLastError();
    if (e == cudaSuccess) {
        sum_partials_kernel<<<1, 32, 0, st>>>(partial, blocks, out);
        e = cudaGetLastError();
    }
    cudaFreeAsync(partial, st);
    if (e != cudaSuccess) return cuda_error(e, "path cost kernel launch");
    return MRPOP_OK;
}

mrpop_status launch_path_cost(const float *path, int64_t M, int dim, double *out,
                              cudaStream_t st) {
    const uintptr_t at = reinterpret_cast<uintptr_t>(path);
    if (dim % 4 == 0 && at % 16 == 0) return path_cost_v<4>(path, M, dim, out, st);
    if (dim % 2 == 0 && at % 8 == 0) return path_cost_v<2>(path, M, dim, out, st);
    return path_cost_v<1>(path, M, dim, out, st);
}

}  // namespace mrpop

namespace mrpop {

// ---------------------------------------------------------------------------
// Allocation-free NEAREST (mrpop_nearest_noalloc).
//
// mrpop_nearest may take stream-ordered scratch for the partial minima of a
// split tree.  Some callers cannot allocate device memory at query time: a
// real-time replanning loop that must neither stall on the allocator nor risk
// an out-of-memory failure in the middle of a control cycle, or a process whose
// device memory has already been reserved by another framework's caching
// allocator.  For them this variant keeps its partial minima in one fixed
// file-scope device array, g_nearest_noalloc_scratch, which every GPU that
// loads this library holds until the process exits.
//
// Host code cannot use the array's name as a device address (it is a host-side
// stand-in), so every call looks the address up with cudaGetSymbolAddress on
// the current device.  The lookup allocates nothing once the module is loaded
// on that device, which the first call on a device (or any earlier call of
// this library there) does; that first call should therefore come before any
// stream capture.  Not caching the address keeps it right after a device reset
// reloads the module at a new address.  All calls share the array;
// two calls that overlap on the GPU (for example on two streams) race on it.
// Every partial record a call reads was written earlier by the same call, so
// nothing needs clearing between calls.
// ---------------------------------------------------------------------------
namespace {

constexpr int kNoAllocRecords = 2 * MRPOP_NEAREST_NOALLOC_MAX_QUERIES;

__device__ __align__(256) Best g_nearest_noalloc_scratch[kNoAllocRecords];

// Device address of the array on the current device (looked up on every call).
mrpop_status noalloc_scratch(Best **out) {
    void *p = nullptr;
    const cudaError_t e = cudaGetSymbolAddress(&p, g_nearest_noalloc_scratch);
    if (e != cudaSuccess) return cuda_error(e, "cudaGetSymbolAddress(nearest scratch)");
    *out = static_cast<Best *>(p);
    return MRPOP_OK;
}

}  // namespace
}  // namespace mrpop

extern "C" mrpop_status mrpop_nearest_noalloc(const float *tree, int64_t N, int64_t ld,
                                              int32_t dim, const float *queries,
                                              const float *budgets, int64_t Q,
                                              int64_t *out_idx, void *stream) {
    using namespace mrpop;
    if (dim < 1 || dim > MRPOP_MAX_LINKS)
        return set_error(MRPOP_EINVAL, "mrpop_nearest_noalloc: dim=%d outside [1, %d]", dim,
                         MRPOP_MAX_LINKS);
    if (N < 0 || Q < 0 || ld < N || N > (int64_t)INT32_MAX)
        return set_error(MRPOP_EINVAL, "mrpop_nearest_noalloc: bad sizes N=%lld ld=%lld Q=%lld",
                         (long long)N, (long long)ld, (long long)Q);
    if (Q > MRPOP_NEAREST_NOALLOC_MAX_QUERIES)
        return set_error(MRPOP_EINVAL,
                         "mrpop_nearest_noalloc: %lld queries exceed the fixed scratch limit of %d "
                         "(MRPOP_NEAREST_NOALLOC_MAX_QUERIES); split the batch or use mrpop_nearest",
                         (long long)Q, MRPOP_NEAREST_NOALLOC_MAX_QUERIES);
    if (Q == 0) return MRPOP_OK;
    if (!queries || !budgets || !out_idx || (N > 0 && !tree))
        return set_error(MRPOP_EINVAL, "mrpop_nearest_noalloc: NULL buffer");
    Best *scratch = nullptr;
    mrpop_status s = noalloc_scratch(&scratch);
    if (s != MRPOP_OK) return s;
    cudaStream_t st = (cudaStream_t)stream;
    const int n = (int)N, q = (int)Q;
    int dev = 0, sms = 1, chunk = 0, splits = 1;
    MRPOP_CUDA_TRY(cudaGetDevice(&dev));
    MRPOP_CUDA_TRY(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
    if (small_scan(dim, n, q, sms, kNoAllocRecords)) {
        small_slices(n, q, sms, kNoAllocRecords, &chunk, &splits);
        return small_dims(tree, n, ld, dim, queries, budgets, q, chunk, splits, out_idx,
                          splits > 1 ? scratch : nullptr, st);
    }
    scan_slices(n, q, sms, kNoAllocRecords, &chunk, &splits);
    bool clusters = true;
    if ((s = scan_in_clusters(splits, q, &clusters)) != MRPOP_OK) return s;
    return scan_rows(tree, n, ld, dim, queries, budgets, q, chunk, splits, out_idx,
                     clusters ? nullptr : scratch, nullptr, st);
}
