// Motion validation of composite edges (Sec. III-E) and forward kinematics.
//
// Design (sm_103a, FP32 SIMT; not a dense contraction, so no tensor cores):
//  * One warp per edge, fetched dynamically from a self-resetting work
//    counter.  The edge's q_a and q_b - q_a are staged in shared memory and the
//    interval count n is computed once per warp.
//  * Checkpoints across lanes: tile t of an edge with n+1 points and
//    T = ceil((n+1)/32) tiles assigns point k = t + T*lane to each lane, so
//    every tile samples the whole edge and a collision anywhere ends the edge
//    after few tiles (early exit with __any_sync).
//  * Per link, forward kinematics in registers (Rz, then the d/a/alpha
//    offsets), then four levels of culling:
//      1. the obstacles' distance field (mrpop_internal.cuh): one byte per
//         checkpoint tells whether the link's coarse sphere is clear of all of
//         them; where every lane is clear nothing below runs;
//      2. tile level: the warp bounds the link's coarse spheres at the near
//         checkpoints by one sphere; lane i tests obstacle i against it, and a
//         ballot gives the candidate set;
//      3. checkpoint level ("coarse" stage of the paper): each lane tests its
//         own link sphere against the candidates only;
//      4. sphere level ("fine" stage): the warp-wide OR of the lanes' hit
//         masks (__reduce_or_sync) selects the obstacles / links whose spheres
//         are tested.
//    Robots are tested against each other through boxes (per tile, then per
//    checkpoint), link spheres, then spheres.
//    The clearance and work-count modes and the reassigned fine stage keep the
//    form without the field (validate_body), which the counters describe.
//    Culling never changes a verdict: each bound encloses what it replaces
//    with a slack above FP32 rounding.
//  * The paper's own design (4 threads per motion, then threads reassigned in
//    proportion to the fine-test load) balances work across motions; here the
//    warp-uniform union mask keeps all 32 lanes busy on the same tests instead.
//  * Geometry tables are staged once per block into shared memory; the links'
//    coarse centres go to a per-warp shared scratch [link][3][lane]
//    (lane-contiguous, conflict-free) for the robot-robot tests, whose rare
//    fine stage rebuilds the links' frames.
#include <cfloat>
#include <cmath>
#include <algorithm>
#include <map>
#include <mutex>
#include <set>
#include <tuple>

#include "mrpop_internal.cuh"
#include "validate_body.cuh"

namespace mrpop {
namespace {

using namespace vb;

template <int MODE, bool RA, bool SHARE = true>
__global__ void __launch_bounds__(kWarpsMax * 32, MODE == kVerdict && !RA ? 7 : 1)
validate_kernel(const __grid_constant__ VParams P) {
    extern __shared__ float4 sm4[];
    if constexpr (MODE == kVerdict && !RA)
        verdict_body<false, false, SHARE>(P, sm4);
    else
        validate_body<MODE, RA>(P, sm4);
}

// One edge per block (few edges).
__global__ void __launch_bounds__(kWarpsMax * 32)
validate_group_kernel(const __grid_constant__ VParams P) {
    extern __shared__ float4 sm4[];
    __shared__ int s_hit;
    if (threadIdx.x == 0) s_hit = 0;  // (visible after the tables' barrier)
    verdict_body<false, true>(P, sm4, 0, 0, &s_hit);
}

// The same kernel with a wide register budget (up to 128 registers: four
// blocks of four warps per SM): fewer warps, no spills in the robot-robot
// fine stage, which many-arm scenes reach often.  An autotuner dimension.
template <int MODE, bool RA, bool SHARE = true>
__global__ void __launch_bounds__(kWarpsMax * 32, 4) validate_kernel_wide(const __grid_constant__ VParams P) {
    extern __shared__ float4 sm4[];
    if constexpr (MODE == kVerdict && !RA)
        verdict_body<false, false, SHARE>(P, sm4);
    else
        validate_body<MODE, RA>(P, sm4);
}

// Many problems in one launch: block row y serves problem y (its parameters
// are staged in shared memory once per block).
template <bool RA>
__global__ void __launch_bounds__(kWarpsMax * 32) validate_batch_kernel(const VParams *Ps) {
    extern __shared__ float4 sm4[];
    __shared__ VParams sP;
    if (threadIdx.x == 0) sP = Ps[blockIdx.y];
    __syncthreads();
    if constexpr (RA)
        validate_body<kVerdict, true>(sP, sm4);
    else
        verdict_body<false>(sP, sm4);
}

// Resident blocks per SM of a validation kernel for a launch shape.  The
// kernel's dynamic shared-memory limit is raised to the device maximum once,
// and occupancies are cached per (kernel, device, threads, bytes): the
// planner issues thousands of small validation launches, and these host
// queries would otherwise cost more than the launches themselves.
static mrpop_status cached_occupancy(const void *kern, int device, int smem_optin, int threads,
                                     size_t smem, int *bps) {
    static std::mutex mu;
    static std::map<std::tuple<const void *, int, int, size_t>, int> occ;
    static std::set<std::pair<const void *, int>> raised;
    std::lock_guard<std::mutex> lock(mu);
    if (!raised.count({kern, device})) {
        cudaFuncAttributes fa{};
        MRPOP_CUDA_TRY(cudaFuncGetAttributes(&fa, kern));
        const int limit = smem_optin - (int)fa.sharedSizeBytes;  // static shared memory counts too
        MRPOP_CUDA_TRY(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                            limit));
        raised.insert({kern, device});
    }
    const auto key = std::make_tuple(kern, device, threads, smem);
    auto it = occ.find(key);
    if (it == occ.end()) {
        int b = 0;
        MRPOP_CUDA_TRY(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&b, kern, threads, smem));
        it = occ.emplace(key, b).first;
    }
    *bps = it->second;
    return MRPOP_OK;
}

// An edge per block, whose warps share its tiles, for up to kGroupWaves times
// the edges whose blocks fit on the chip at once (table pair: 1,500 edges 33.8
// us with an edge per warp, 26.5 so; 3,000 edges 39.9 and 42.6).
constexpr int64_t kGroupWaves = 2;
// Above that a warp takes an edge, and warps that find none left help the
// others (SHARE), unless the claims cost more than the tail that they shorten:
// with few links, whose tiles are short (planar pair, 6 links: 8,000 edges 35.4
// us shared, 33.6 not; 65,536 edges 165 and 140), and with many edges for each
// resident warp (table pair, 14 links, 4,256 warps: 8,000 edges 56 us shared,
// 66 not; 16,000 edges 80 and 83; 32,768 edges 136 and 134; 65,536 edges 247
// and 237).
constexpr int kShareLinks = 10;
constexpr int64_t kShareWaves = 6;

template <int MODE, bool RA>
mrpop_status launch_mode(mrpop_problem *p, VParams &V, int warps, size_t smem,
                         cudaStream_t st) {
    auto kern = MODE == kVerdict && p->tuned_regs ? validate_kernel_wide<MODE, RA>
                                                  : validate_kernel<MODE, RA>;
    int bps = 0;
    const mrpop_status os = cached_occupancy((const void *)kern, p->device, (int)p->smem_optin,
                                             warps * 32, smem, &bps);
    if (os != MRPOP_OK) return os;
    if (bps < 1) return set_error(MRPOP_EINVAL, "validation kernel does not fit on an SM");
    // few edges: 256 planar edges 12.3 us (ncu, cold L2), 18.0 with an edge per warp
    if (MODE == kVerdict && !RA && warps > 1 && V.E <= kGroupWaves * p->num_sms * bps) {
        int gbps = 0;
        const mrpop_status gs = cached_occupancy((const void *)validate_group_kernel, p->device,
                                                 (int)p->smem_optin, warps * 32, smem, &gbps);
        if (gs != MRPOP_OK) return gs;
        if (V.E <= kGroupWaves * p->num_sms * gbps) {
            V.warps = warps;
            validate_group_kernel<<<(int)V.E, warps * 32, smem, st>>>(V);
            MRPOP_CUDA_TRY(cudaGetLastError());
            return MRPOP_OK;
        }
    }
    if constexpr (MODE == kVerdict && !RA) {
        const int64_t shared_warps = (int64_t)p->num_sms * bps * warps;
        if (V.t.L < kShareLinks || V.E > kShareWaves * shared_warps) {
            // a kernel of its own, with its own shared-memory limit and occupancy
            kern = p->tuned_regs ? validate_kernel_wide<MODE, RA, false>
                                 : validate_kernel<MODE, RA, false>;
            const mrpop_status us = cached_occupancy((const void *)kern, p->device,
                                                     (int)p->smem_optin, warps * 32, smem, &bps);
            if (us != MRPOP_OK) return us;
            if (bps < 1) return set_error(MRPOP_EINVAL, "validation kernel does not fit on an SM");
        }
    }
    const int64_t want = (V.E + warps - 1) / warps;
    const int grid = (int)std::min<int64_t>((int64_t)p->num_sms * bps, want);
    V.total_warps = grid * warps;
    V.warps = warps;
    kern<<<grid, warps * 32, smem, st>>>(V);
    MRPOP_CUDA_TRY(cudaGetLastError());
    return MRPOP_OK;
}

// The reassigned fine stage exists for verdicts only; the clearance and
// work-count modes always take the union form.
template <int MODE>
mrpop_status launch_spl(mrpop_problem *p, VParams &V, int warps, size_t smem,
                        cudaStream_t st) {
    if (MODE == kVerdict && V.fine) return launch_mode<MODE, true>(p, V, warps, smem, st);
    return launch_mode<MODE, false>(p, V, warps, smem, st);
}

// ---------------------------------------------------------------------------
// Forward kinematics of a batch of configurations: one thread per
// configuration and robot (blockIdx.y), the robot's table rows in shared
// memory.  Bound by the stores of the sphere centres, 12 bytes a sphere: read
// from global memory link by link and sphere by sphere, the table's latency
// was most of the time (20,001 configurations of two 60-sphere arms, 29 MB, which
// need 4.4 us: 24.7 us so, 9.8 here (ncu, cold L2); a call 22.5 and 15.8 to 18.5,
// the host's).
// ---------------------------------------------------------------------------
constexpr int kFkThreads = 128;

__global__ void __launch_bounds__(kFkThreads)
fk_kernel(const float4 *__restrict__ tab, const __grid_constant__ Tables t,
          const float *__restrict__ q, int64_t n, float *__restrict__ out) {
    // base (3), then (a, d, cos alpha, sin alpha) and (theta_offset, first
    // sphere, count, -) of each link, then the link's spheres
    __shared__ float4 sm[3 + 2 * MRPOP_MAX_DOF + MRPOP_MAX_DOF * MRPOP_MAX_SPHERES_PER_LINK];
    const int b = blockIdx.y, l0 = t.link0[b], dof = t.link0[b + 1] - l0;
    float4 *lk = sm + 3, *sp = lk + 2 * MRPOP_MAX_DOF;
    const float4 *first = tab + t.off_link + kLinkF4 * l0;
    const float4 *last = first + kLinkF4 * (dof - 1);
    const int s0 = __float_as_int(__ldg(first + 1).y);
    const float4 lb = __ldg(last + 1);
    const int ns_all = __float_as_int(lb.y) + __float_as_int(lb.z) - s0;
    if (threadIdx.x < 3) sm[threadIdx.x] = __ldg(tab + t.off_base + 3 * b + threadIdx.x);
    for (int i = threadIdx.x; i < 2 * dof; i += kFkThreads)
        lk[i] = __ldg(first + kLinkF4 * (i >> 1) + (i & 1));
    for (int i = threadIdx.x; i < ns_all; i += kFkThreads) sp[i] = __ldg(tab + t.off_sph + s0 + i);
    __syncthreads();
    const int64_t i = (int64_t)blockIdx.x * kFkThreads + threadIdx.x;
    if (i >= n) return;
    const int64_t S = t.S;
    Frame Tm;
    const float4 r0 = sm[0], r1 = sm[1], r2 = sm[2];
    Tm.r[0] = r0.x; Tm.r[1] = r0.y; Tm.r[2] = r0.z; Tm.t[0] = r0.w;
    Tm.r[3] = r1.x; Tm.r[4] = r1.y; Tm.r[5] = r1.z; Tm.t[1] = r1.w;
    Tm.r[6] = r2.x; Tm.r[7] = r2.y; Tm.r[8] = r2.z; Tm.t[2] = r2.w;
    const float *qi = q + (size_t)l0 * n + i;
    float *ox = out + (size_t)s0 * n + i, *oy = ox + (size_t)S * n, *oz = oy + (size_t)S * n;
    float th = __ldg(qi);
    for (int j = 0; j < dof; ++j) {
        const float4 LA = lk[2 * j], LB = lk[2 * j + 1];
        float sn, cs;
        joint_sincos(th + LB.x, &sn, &cs);
        qi += n;
        if (j + 1 < dof) th = __ldg(qi);
        const Frame F = rotz(Tm, cs, sn);
        const int ns = __float_as_int(LB.z);
#pragma unroll 4
        for (int s = 0; s < ns; ++s) {
            const float4 c = *sp++;
            const float3 pw = apply(F, c.x, c.y, c.z);
            *ox = pw.x;
            *oy = pw.y;
            *oz = pw.z;
            ox += n;
            oy += n;
            oz += n;
        }
        Tm = advance(F, LA.x, LA.y, LA.z, LA.w);
    }
}

// Distance field of the obstacles, one voxel per thread (DistanceField in
// mrpop_internal.cuh).  Bound by the obstacle tests (11 flops a sphere, 31 a
// box), once per problem: 229,000 voxels and 64 obstacles on the table pair;
// problem creation grew by about 0.12 ms with the field's allocation.
__global__ void __launch_bounds__(256)
field_kernel(const float4 *__restrict__ tab, const Tables t, float edge, float shrink, float unit,
             uint8_t *__restrict__ out) {
    const int nx = t.df_n[0], ny = t.df_n[1], nz = t.df_n[2];
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= nx * ny * nz) return;
    const int ix = i % nx, iy = (i / nx) % ny, iz = i / (nx * ny);
    const float x = edge * (kFieldMagic - t.df_c[0] + (float)ix);
    const float y = edge * (kFieldMagic - t.df_c[1] + (float)iy);
    const float z = edge * (kFieldMagic - t.df_c[2] + (float)iz);
    float d = FLT_MAX;
    for (int o = 0; o < t.NS; ++o) {
        const float4 ob = __ldg(tab + t.off_os + o);
        d = fminf(d, __fsqrt_rn(dist2(x, y, z, ob.x, ob.y, ob.z)) - ob.w);
    }
    float d2 = FLT_MAX;
    for (int o = 0; o < t.NC; ++o) {
        const float4 *c = tab + t.off_oc + kCuboidF4 * o;
        d2 = fminf(d2, box_dist2(x, y, z, __ldg(c), __ldg(c + 1), __ldg(c + 2), __ldg(c + 3),
                                 __ldg(c + 4)));
    }
    d = fminf(d, __fsqrt_rn(d2)) - shrink;
    // (a NaN bound, which finite tables do not give, reads as near)
    out[i] = d > 0.f ? (uint8_t)fminf(255.f, floorf(d / unit * 0.99999f)) : 0;
}

}  // namespace

mrpop_status launch_field(const Tables &t, const float4 *blob, float edge, float shrink, float unit,
                          uint8_t *out, cudaStream_t st) {
    const int n = t.df_n[0] * t.df_n[1] * t.df_n[2];
    field_kernel<<<(n + 255) / 256, 256, 0, st>>>(blob, t, edge, shrink, unit, out);
    MRPOP_CUDA_TRY(cudaGetLastError());
    return MRPOP_OK;
}

mrpop_status launch_validate(mrpop_problem *p, const float *qa, const float *qb, int64_t n,
                             uint8_t *valid, float *length, int32_t *npoints,
                             float *min_clear, unsigned long long *counters,
                             cudaStream_t st) {
    const Tables &t = p->dev.t;
    VParams V;
    V.t = t;
    V.blob = p->dev.blob;
    V.qa = qa;
    V.qb = qb;
    V.E = n;
    V.res = p->cfg.resolution;
    V.margin = p->cfg.margin;
    V.valid = valid;
    V.length = length;
    V.npoints = npoints;
    V.min_clear = min_clear;
    V.counters = counters;
    V.work = p->dev.edge_counter;
    V.dpad = (t.L + 3) & ~3;
    V.nstore = t.selfcol ? t.L : t.link0[t.K - 1];
    V.fine = p->tuned_fine;
    V.warp_floats = min_clear || counters || V.fine ? validate_warp_floats(t, V.fine)
                                                    : verdict_warp_floats(t);
    const size_t tab_bytes = (size_t)t.n_f4 * sizeof(float4);
    int warps = p->tuned_warps > 0 ? p->tuned_warps : kWarpsMax;
    size_t smem = 0;
    for (; warps >= 1; warps >>= 1) {
        smem = tab_bytes + (size_t)warps * V.warp_floats * sizeof(float);
        if (smem <= p->smem_optin) break;
    }
    V.order = p->tuned_order;
    if (warps < 1)
        return set_error(MRPOP_EINVAL,
                         "problem too large for the validation kernel's shared memory "
                         "(%zu bytes of tables + %d bytes per warp)",
                         tab_bytes, V.warp_floats * 4);
    if (min_clear) return launch_spl<kClearance>(p, V, warps, smem, st);
    if (counters) return launch_spl<kCount>(p, V, warps, smem, st);
    return launch_spl<kVerdict>(p, V, warps, smem, st);
}

mrpop_status make_vparams(mrpop_problem *p, const float *qa, const float *qb, int64_t n,
                          uint8_t *valid, VParams *V, size_t *smem_out, int *warps_out) {
    const Tables &t = p->dev.t;
    *V = VParams{};
    V->t = t;
    V->blob = p->dev.blob;
    V->qa = qa;
    V->qb = qb;
    V->E = n;
    V->res = p->cfg.resolution;
    V->margin = p->cfg.margin;
    V->valid = valid;
    V->work = p->dev.edge_counter;
    V->dpad = (t.L + 3) & ~3;
    V->nstore = t.selfcol ? t.L : t.link0[t.K - 1];
    V->fine = p->tuned_fine;
    // (a slot that asks for the reassigned stage may share a launch without it)
    V->warp_floats = std::max(verdict_warp_floats(t), V->fine ? validate_warp_floats(t, 1) : 0);
    const size_t tab_bytes = (size_t)t.n_f4 * sizeof(float4);
    int warps = p->tuned_warps > 0 ? p->tuned_warps : kWarpsMax;
    size_t smem = 0;
    for (; warps >= 1; warps >>= 1) {
        smem = tab_bytes + (size_t)warps * V->warp_floats * sizeof(float);
        if (smem + sizeof(VParams) + 1024 <= p->smem_optin) break;
    }
    V->order = p->tuned_order;
    if (warps < 1)
        return set_error(MRPOP_EINVAL, "problem too large for the validation kernel's shared memory");
    *smem_out = smem;
    *warps_out = warps;
    V->warps = warps;
    return MRPOP_OK;
}

template <bool RA>
static mrpop_status batch_ra(const VParams *d_params, int nslots, int warps, int blocks_per_slot,
                             size_t smem, cudaStream_t st) {
    auto kern = validate_batch_kernel<RA>;
    int dev = 0, optin = 0, bps = 0;
    MRPOP_CUDA_TRY(cudaGetDevice(&dev));
    MRPOP_CUDA_TRY(cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev));
    const mrpop_status os = cached_occupancy((const void *)kern, dev, optin, warps * 32, smem, &bps);
    if (os != MRPOP_OK) return os;
    dim3 grid(blocks_per_slot, nslots);
    kern<<<grid, warps * 32, smem, st>>>(d_params);
    MRPOP_CUDA_TRY(cudaGetLastError());
    return MRPOP_OK;
}

mrpop_status launch_validate_batch(const VParams *d_params, int nslots, int /*spl*/, int warps,
                                   int blocks_per_slot, size_t smem, bool fine,
                                   cudaStream_t st) {
    if (fine) return batch_ra<true>(d_params, nslots, warps, blocks_per_slot, smem, st);
    return batch_ra<false>(d_params, nslots, warps, blocks_per_slot, smem, st);
}

// Times the validation kernel on the caller's edges for every candidate
// launch (warps per block 1, 2, 4 that fit; strided or contiguous checkpoint
// order; union or reassigned fine tests; compact or wide register budget),
// keeps the fastest in the problem and in the tuned-launch cache under the
// problem's shape, and reports it.
mrpop_status autotune_validate(mrpop_problem *p, const float *qa, const float *qb, int64_t n,
                               uint8_t *valid, int reps, int32_t *out, float *ms_out,
                               cudaStream_t st) {
    cudaEvent_t a, b;
    MRPOP_CUDA_TRY(cudaEventCreate(&a));
    MRPOP_CUDA_TRY(cudaEventCreate(&b));
    float best = INFINITY;
    int bw = 0, bo = 0, bf = 0, br = 0;
    const int save_w = p->tuned_warps, save_o = p->tuned_order, save_f = p->tuned_fine,
              save_r = p->tuned_regs;
    mrpop_status s = MRPOP_OK;
    for (int w = 1; w <= kWarpsMax && s == MRPOP_OK; w *= 2)
        for (int o = 0; o < 2 && s == MRPOP_OK; ++o)
        for (int f = 0; f < 2 && s == MRPOP_OK; ++f)
        for (int rg = 0; rg < 2 && s == MRPOP_OK; ++rg) {
            const size_t need = (size_t)p->dev.t.n_f4 * sizeof(float4) +
                                (size_t)w * sizeof(float) *
                                    std::max(verdict_warp_floats(p->dev.t),
                                             f ? validate_warp_floats(p->dev.t, 1) : 0);
            if (need + sizeof(VParams) + 1024 > p->smem_optin) continue;
            p->tuned_warps = w;
            p->tuned_order = o;
            p->tuned_fine = f;
            p->tuned_regs = rg;
            s = launch_validate(p, qa, qb, n, valid, nullptr, nullptr, nullptr, nullptr, st);  // warm
            float tot = 0.f;
            for (int r = 0; r < reps && s == MRPOP_OK; ++r) {
                cudaEventRecord(a, st);
                s = launch_validate(p, qa, qb, n, valid, nullptr, nullptr, nullptr, nullptr, st);
                cudaEventRecord(b, st);
                cudaEventSynchronize(b);
                float ms = 0.f;
                cudaEventElapsedTime(&ms, a, b);
                tot += ms;
            }
            if (s == MRPOP_OK && tot < best) {
                best = tot;
                bw = w;
                bo = o;
                bf = f;
                br = rg;
            }
        }
    cudaEventDestroy(a);
    cudaEventDestroy(b);
    if (s != MRPOP_OK || bw == 0) {
        p->tuned_warps = save_w;
        p->tuned_order = save_o;
        p->tuned_fine = save_f;
        p->tuned_regs = save_r;
        return s != MRPOP_OK ? s : set_error(MRPOP_EINVAL, "no launch configuration fits");
    }
    p->tuned_warps = bw;
    p->tuned_order = bo;
    p->tuned_fine = bf;
    p->tuned_regs = br;
    tune_store(validate_tune_key(p), {bw, bo, bf, br});
    if (out) {
        out[0] = bw;
        out[1] = bo;
        out[2] = bf;
    }
    if (ms_out) *ms_out = best / std::max(1, reps);
    return MRPOP_OK;
}

mrpop_status launch_fk(mrpop_problem *p, const float *q, int64_t n, float *out, cudaStream_t st) {
    const int64_t blocks = (n + kFkThreads - 1) / kFkThreads;
    fk_kernel<<<dim3((unsigned)blocks, p->dev.t.K), kFkThreads, 0, st>>>(p->dev.blob, p->dev.t, q, n,
                                                                         out);
    MRPOP_CUDA_TRY(cudaGetLastError());
    return MRPOP_OK;
}

}  // namespace mrpop
