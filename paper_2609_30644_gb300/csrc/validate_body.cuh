// Validation body shared by the validation kernels (validate.cu) and the
// planner's persistent kernel (planner.cu): one warp per edge, checkpoints
// across lanes, per-link FK with tile / checkpoint / sphere culling and
// early exit.  See validate.cu for the design.
#pragma once
#include <cfloat>

#include "mrpop_internal.cuh"

namespace mrpop {
namespace vb {

constexpr unsigned kFull = 0xffffffffu;
constexpr int kWarpsMax = 4;
constexpr int kCounters = MRPOP_WORK_COUNTERS;
// Absolute slack (m) added to tile bounds: covers FP32 rounding of the box
// centre and half extents (a few ulps of workspace coordinates), so the tile
// test never drops a candidate that a checkpoint's own link-level test keeps.
constexpr float kTileSlack = 4e-4f;


enum Mode { kVerdict = 0, kClearance = 1, kCount = 2 };



struct Frame {
    float r[9];  // row-major rotation
    float t[3];
};

// F = T * Rz(theta): columns 0 and 1 rotate, column 2 and t are unchanged.
__device__ __forceinline__ Frame rotz(const Frame &T, float c, float s) {
    Frame F;
#pragma unroll
    for (int i = 0; i < 3; ++i) {
        const float a = T.r[3 * i], b = T.r[3 * i + 1];
        F.r[3 * i] = fmaf(c, a, s * b);
        F.r[3 * i + 1] = fmaf(c, b, -s * a);
        F.r[3 * i + 2] = T.r[3 * i + 2];
        F.t[i] = T.t[i];
    }
    return F;
}

// T = F * Tz(d) * Tx(a) * Rx(alpha)
__device__ __forceinline__ Frame advance(const Frame &F, float a, float d, float ca, float sa) {
    Frame T;
#pragma unroll
    for (int i = 0; i < 3; ++i) {
        const float c0 = F.r[3 * i], c1 = F.r[3 * i + 1], c2 = F.r[3 * i + 2];
        T.t[i] = fmaf(a, c0, fmaf(d, c2, F.t[i]));
        T.r[3 * i] = c0;
        T.r[3 * i + 1] = fmaf(ca, c1, sa * c2);
        T.r[3 * i + 2] = fmaf(ca, c2, -sa * c1);
    }
    return T;
}

__device__ __forceinline__ float3 apply(const Frame &F, float x, float y, float z) {
    return make_float3(fmaf(F.r[0], x, fmaf(F.r[1], y, fmaf(F.r[2], z, F.t[0]))),
                       fmaf(F.r[3], x, fmaf(F.r[4], y, fmaf(F.r[5], z, F.t[1]))),
                       fmaf(F.r[6], x, fmaf(F.r[7], y, fmaf(F.r[8], z, F.t[2]))));
}

__device__ __forceinline__ float dist2(float ax, float ay, float az, float bx, float by,
                                       float bz) {
    const float dx = ax - bx, dy = ay - by, dz = az - bz;
    return fmaf(dx, dx, fmaf(dy, dy, dz * dz));
}

// Squared distance from point p to an oriented box (centre C, half extents H,
// unit axes A0..A2 as columns): |max(|A^T (p - C)| - h, 0)|^2.
__device__ __forceinline__ float box_dist2(float px, float py, float pz, const float4 &C,
                                           const float4 &H, const float4 &A0, const float4 &A1,
                                           const float4 &A2) {
    const float vx = px - C.x, vy = py - C.y, vz = pz - C.z;
    const float p0 = fmaf(A0.x, vx, fmaf(A0.y, vy, A0.z * vz));
    const float p1 = fmaf(A1.x, vx, fmaf(A1.y, vy, A1.z * vz));
    const float p2 = fmaf(A2.x, vx, fmaf(A2.y, vy, A2.z * vz));
    const float u0 = fmaxf(fabsf(p0) - H.x, 0.f);
    const float u1 = fmaxf(fabsf(p1) - H.y, 0.f);
    const float u2 = fmaxf(fabsf(p2) - H.z, 0.f);
    return fmaf(u0, u0, fmaf(u1, u1, u2 * u2));
}

__device__ __forceinline__ Frame load_base(const float4 *tab, const Tables &t, int b) {
    const float4 r0 = tab[t.off_base + 3 * b], r1 = tab[t.off_base + 3 * b + 1],
                 r2 = tab[t.off_base + 3 * b + 2];
    Frame T;
    T.r[0] = r0.x; T.r[1] = r0.y; T.r[2] = r0.z; T.t[0] = r0.w;
    T.r[3] = r1.x; T.r[4] = r1.y; T.r[5] = r1.z; T.t[1] = r1.w;
    T.r[6] = r2.x; T.r[7] = r2.y; T.r[8] = r2.z; T.t[2] = r2.w;
    return T;
}

// Frame F_i' of link i at the lane's checkpoint (parameter tk), rebuilt along
// its robot's chain from the base with the same operations, in the same order,
// as the main forward-kinematics loop.  Used only by fine robot-robot tests,
// which are rare; the coarse tests read the stored coarse centres.
__device__ __forceinline__ Frame link_frame(const float4 *tab, const Tables &t, const float *qa_s,
                                            const float *dq_s, int i, float tk);

// Joint-angle sine and cosine: reduce the angle to [-pi, pi] with one fused
// multiply-add, then the hardware approximation __sincosf (absolute error
// about 2^-21 on that interval; over a 7-joint chain with a 1.2 m reach it
// moves a sphere by a few micrometres, far inside the 1e-4 m contact band
// and the 1e-5 relative distance tolerance).
__device__ __forceinline__ void joint_sincos(float th, float *s, float *c) {
    const float k = rintf(th * 0.15915494f);        // th / (2 pi), nearest integer
    __sincosf(fmaf(-6.28318548f, k, th), s, c);
}

// Smallest of the warp's values (order-preserving integer keys; no NaN).
__device__ __forceinline__ float warp_min(float v) {
    const int k = __float_as_int(v);
    const int r = __reduce_min_sync(kFull, k ^ ((k >> 31) & 0x7fffffff));
    return __int_as_float(r ^ ((r >> 31) & 0x7fffffff));
}

// Second stage with load-proportional reassignment (Sec. III-E): the fine
// tests that the lanes' own coarse hits call for -- (checkpoint k, obstacle o
// hit by k's link sphere, fine sphere s of the link) -- are numbered by a warp
// prefix sum of the per-lane counts and dealt out to all 32 lanes in turn, so
// the warp spends ceil(total / 32) passes on them instead of one pass of
// every lane over every obstacle that any lane hit.  A lane rebuilds its
// item's fine sphere from the owning checkpoint's link frame, which every lane
// puts in the warp's shared scratch fr ([12][32] floats, then 32 hit masks and
// 32 prefix sums).  A fine hit implies a coarse hit (the coarse sphere encloses
// the fine ones with slack), so the verdict equals the union form's.
template <bool CUBOID>
__device__ __forceinline__ bool fine_reassigned(unsigned own, int c0, int ns, int sf,
                                                const Frame &F, float m, const float4 *tab,
                                                const Tables &t, float *fr, int lane) {
    if (!__any_sync(kFull, own != 0u)) return false;  // the common case: no fine work
    const int mine = __popc(own) * ns;
    int incl = mine;
#pragma unroll
    for (int off = 1; off < 32; off <<= 1) {
        const int y = __shfl_up_sync(kFull, incl, off);
        if (lane >= off) incl += y;
    }
    const int total = __shfl_sync(kFull, incl, 31);
    if (total == 0) return false;
    unsigned *own_s = reinterpret_cast<unsigned *>(fr + kFrFloats * 32);
    int *pre_s = reinterpret_cast<int *>(own_s + 32);
#pragma unroll
    for (int c = 0; c < 9; ++c) fr[c * 32 + lane] = F.r[c];
    fr[9 * 32 + lane] = F.t[0];
    fr[10 * 32 + lane] = F.t[1];
    fr[11 * 32 + lane] = F.t[2];
    own_s[lane] = own;
    pre_s[lane] = incl - mine;
    __syncwarp();
    const float inv_ns = 1.f / (float)ns;
    bool hit = false;
    for (int b = 0; b < total; b += 32) {
        const int item = b + lane;
        if (item < total) {
            int k = 0;  // owner: the last lane whose first item is <= item
#pragma unroll
            for (int step = 16; step > 0; step >>= 1)
                if (pre_s[k + step] <= item) k += step;
            const int r = item - pre_s[k];
            int jo = (int)((float)r * inv_ns);  // r / ns, corrected below
            if (jo * ns > r) --jo;
            if ((jo + 1) * ns <= r) ++jo;
            const int s = r - jo * ns;
            unsigned mm = own_s[k];
            for (int q = 0; q < jo; ++q) mm &= mm - 1;  // jo-th set bit of k's mask
            const int o = __ffs(mm) - 1;
            Frame Fk;
#pragma unroll
            for (int c = 0; c < 9; ++c) Fk.r[c] = fr[c * 32 + k];
            Fk.t[0] = fr[9 * 32 + k];
            Fk.t[1] = fr[10 * 32 + k];
            Fk.t[2] = fr[11 * 32 + k];
            const float4 sp = tab[t.off_sph + sf + s];
            const float3 p = apply(Fk, sp.x, sp.y, sp.z);
            if (CUBOID) {
                const float4 *cbp = tab + t.off_oc + kCuboidF4 * (c0 + o);
                const float d2 = box_dist2(p.x, p.y, p.z, cbp[0], cbp[1], cbp[2], cbp[3], cbp[4]);
                const float th2 = sp.w + m;
                hit |= d2 < th2 * th2;
            } else {
                const float4 ob = tab[t.off_os + c0 + o];
                const float d2 = dist2(p.x, p.y, p.z, ob.x, ob.y, ob.z);
                const float th2 = sp.w + ob.w + m;
                hit |= d2 < th2 * th2;
            }
        }
    }
    __syncwarp();  // the scratch is rewritten by the next call
    return hit;
}

__device__ __forceinline__ Frame link_frame(const float4 *tab, const Tables &t, const float *qa_s,
                                            const float *dq_s, int i, float tk) {
    int b = 0;
    while (t.link0[b + 1] <= i) ++b;
    Frame Tm = load_base(tab, t, b);
    for (int l = t.link0[b];; ++l) {
        const float4 LA = tab[t.off_link + kLinkF4 * l];
        const float4 LB = tab[t.off_link + kLinkF4 * l + 1];
        const float th = __fmaf_rn(tk, dq_s[l], qa_s[l]) + LB.x;
        float sn, cs;
        joint_sincos(th, &sn, &cs);
        const Frame F = rotz(Tm, cs, sn);
        if (l == i) return F;
        Tm = advance(F, LA.x, LA.y, LA.z, LA.w);
    }
}

// Interval count n = max(1, ceil(|dq|_2 / res)) in FP32 with a sequential
// fused multiply-add sum (the oracle takes the same integer decision in FP32).
__device__ __forceinline__ int interval_count(const float *dq, int D, float res, float *len_out) {
    float acc = 0.f;
    for (int i = 0; i < D; ++i) acc = __fmaf_rn(dq[i], dq[i], acc);
    const float len = __fsqrt_rn(acc);
    const float nf = ceilf(__fdiv_rn(len, res));
    *len_out = len;
    if (!(nf >= 1.f)) return 1;
    return nf > 1073741824.f ? 1073741824 : (int)nf;
}

// The clearance and work-count modes, and verdicts with the reassigned fine
// stage.  Clearance takes the same levels with a bound from above on the edge's
// minimum clearance in the margin's place: far sides of tile bounds at first,
// then the values themselves, shared by the warp.  A pair that some level
// leaves out lies farther apart than a pair that is measured (every bound
// encloses what it replaces with at least 1e-4 m of slack), so the minimum is
// that over all pairs, to the bit.  Measuring every pair, with a square root
// each, took 2,929 us for 1,023 edges of the table pair; this takes 90 us.
template <int MODE, bool RA>
__device__ __forceinline__ void validate_body(const VParams &P, float4 *sm4) {
    static_assert(MODE != kVerdict || RA, "plain verdicts take verdict_body");
    float4 *tab = sm4;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    float *ws = reinterpret_cast<float *>(sm4 + P.t.n_f4) + (size_t)warp * P.warp_floats;
    float *qa_s = ws, *dq_s = ws + P.dpad;
    float4 *tb = reinterpret_cast<float4 *>(ws + 2 * P.dpad);      // tile bounds [nstore]
    float *xc = ws + 2 * P.dpad + 4 * P.nstore;                     // [nstore][3][32]
    float *fr = xc + P.nstore * kXcFloats * 32;                     // reassignment scratch
    constexpr bool ra = MODE == kVerdict && RA;  // reassigned fine obstacle tests

    for (int i = threadIdx.x; i < P.t.n_f4; i += blockDim.x) tab[i] = P.blob[i];
    __syncthreads();
    if (warp >= P.warps) return;  // spare warps of a shared multi-problem launch

    const Tables &t = P.t;
    // table offsets and the workspace corner read once (the loops below would
    // otherwise reload them from the launch parameters at every use)
    const int o_link = t.off_link, o_os = t.off_os, o_oc = t.off_oc, o_sph = t.off_sph;
    const float wlx = t.ws_lo[0], wly = t.ws_lo[1], wlz = t.ws_lo[2];
    const int K = t.K, D = t.L, NS = t.NS, NC = t.NC;
    const float margin = P.margin;
    unsigned long long cnt[kCounters];
#pragma unroll
    for (int c = 0; c < kCounters; ++c) cnt[c] = 0ull;

    for (;;) {
        int e = 0;
        if (lane == 0) e = atomicAdd(&P.work[0], 1);
        e = __shfl_sync(kFull, e, 0);
        if (e >= P.E) break;
        __syncwarp();
        for (int i = lane; i < D; i += 32) {
            const float a = __ldg(P.qa + (size_t)i * P.E + e);
            const float b = __ldg(P.qb + (size_t)i * P.E + e);
            qa_s[i] = a;
            dq_s[i] = __fsub_rn(b, a);
        }
        __syncwarp();
        float len;
        const int n = interval_count(dq_s, D, P.res, &len);
        // Edges beyond MRPOP_MAX_EDGE_INTERVALS intervals (or with non-finite
        // coordinates) are reported invalid without being checked.
        const bool too_long = !(len <= P.res * (float)MRPOP_MAX_EDGE_INTERVALS);
        const int T = too_long ? 0 : (n >> 5) + 1;  // ceil((n + 1) / 32)
        bool edge_hit = too_long;
        float minc = too_long ? -FLT_MAX : FLT_MAX;
        // kClearance: a bound from above on the edge's minimum clearance
        // (warp-uniform); pairs that lie at least this far apart are skipped
        float m = MODE == kClearance ? FLT_MAX : margin;

        for (int tile = 0; tile < T; ++tile) {
            int k = P.order ? tile * 32 + lane : tile + T * lane;
            const bool active = k <= n;
            if (!active) k = n;
            const float tk = __fdiv_rn((float)k, (float)n);
            bool hit = false;
            if (MODE == kCount && active) cnt[0] += 1;
            // joint angles' sine and cosine one link ahead, so that the
            // special-function latency overlaps the previous link's tests
            float sn_next, cs_next;
            joint_sincos(__fmaf_rn(tk, dq_s[0], qa_s[0]) + tab[o_link + 1].x, &sn_next,
                         &cs_next);

            for (int b = 0; b < K; ++b) {
                const int l0 = t.link0[b], l1 = t.link0[b + 1];
                const bool store = b < K - 1 || t.selfcol;
                Frame Tm = load_base(tab, t, b);
                for (int l = l0; l < l1; ++l) {
                    const float4 LA = tab[o_link + kLinkF4 * l];
                    const float4 LB = tab[o_link + kLinkF4 * l + 1];
                    const float4 LC = tab[o_link + kLinkF4 * l + 2];
                    const float sn = sn_next, cs = cs_next;
                    if (l + 1 < D)
                        joint_sincos(__fmaf_rn(tk, dq_s[l + 1], qa_s[l + 1]) +
                                         tab[o_link + kLinkF4 * (l + 1) + 1].x,
                                     &sn_next, &cs_next);
                    const Frame F = rotz(Tm, cs, sn);
                    const float3 cc = apply(F, LC.x, LC.y, LC.z);
                    const int sf = __float_as_int(LB.y), ns = __float_as_int(LB.z);
                    if (MODE == kCount && active) cnt[1] += 1;

                    // Tile bound: one sphere around this link's coarse spheres at
                    // all 32 checkpoints of the tile (warp-uniform), built from the
                    // exact axis-aligned box of the coarse centres.  Taken relative
                    // to the workspace corner ws_lo the coordinates are >= 0, so
                    // their float bits order like unsigned integers and min and max
                    // are single-instruction warp reductions.
                    float4 bnd = make_float4(0.f, 0.f, 0.f, 0.f);
                    {
                        const unsigned ux = __float_as_uint(cc.x - wlx);
                        const unsigned uy = __float_as_uint(cc.y - wly);
                        const unsigned uz = __float_as_uint(cc.z - wlz);
                        const float x0 = __uint_as_float(__reduce_min_sync(kFull, ux));
                        const float x1 = __uint_as_float(__reduce_max_sync(kFull, ux));
                        const float y0 = __uint_as_float(__reduce_min_sync(kFull, uy));
                        const float y1 = __uint_as_float(__reduce_max_sync(kFull, uy));
                        const float z0 = __uint_as_float(__reduce_min_sync(kFull, uz));
                        const float z1 = __uint_as_float(__reduce_max_sync(kFull, uz));
                        const float ex = 0.5f * (x1 - x0), ey = 0.5f * (y1 - y0),
                                    ez = 0.5f * (z1 - z0);
                        bnd.x = wlx + 0.5f * (x0 + x1);
                        bnd.y = wly + 0.5f * (y0 + y1);
                        bnd.z = wlz + 0.5f * (z0 + z1);
                        // the hardware's approximate square root (an error of a few
                        // ulps), padded by 2^-16 relative; kTileSlack covers the rest
                        float rbox;
                        asm("sqrt.approx.f32 %0, %1;"
                            : "=f"(rbox)
                            : "f"(fmaf(ex, ex, fmaf(ey, ey, ez * ez))));
                        bnd.w = fmaf(rbox, 1.0000153f, LC.w + kTileSlack);
                        if (!(bnd.w < FLT_MAX)) bnd.w = FLT_MAX * 2.f;  // never for finite inputs
                        if (MODE == kCount && lane == 0) cnt[9] += 1;
                    }
                    if (store) {
                        float *x = xc + (size_t)l * kXcFloats * 32 + lane;
                        x[0] = cc.x;
                        x[32] = cc.y;
                        x[64] = cc.z;
                        if (lane == 0) tb[l] = bnd;
                        __syncwarp();
                    }
                    bool vote = false;  // a fine stage ran: the early-exit vote is due
                    // squared distance within reach (clearance: the bound may be
                    // negative, and a reach that is not positive has no pair)
                    auto within = [](float d2, float th) {
                        return MODE == kClearance ? th > 0.f && d2 < th * th : d2 < th * th;
                    };
                    // kClearance: the lanes' minima and new bounds become the warp's
                    auto tighten = [&](float ub) {
                        m = fminf(m, warp_min(fminf(minc, ub)));
                    };
                    if (ns > 0) {
                        bool own_any = false;
                        if (MODE == kCount && active) cnt[7] += 1;  // coarse centre
                        float rc = LC.w + m;

                        // ---- robot vs obstacle spheres
                        for (int c0 = 0; c0 < NS; c0 += 32) {
                            const int cn = min(32, NS - c0);
                            unsigned own = 0, cand = 0;
                            {
                                bool h = false;
                                if (MODE == kClearance) {
                                    // some sphere of the link at some checkpoint is
                                    // within the tile bound's far side of obstacle i
                                    float ub = FLT_MAX;
                                    if (lane < cn) {
                                        const float4 ob = tab[o_os + c0 + lane];
                                        ub = __fsqrt_rn(dist2(bnd.x, bnd.y, bnd.z, ob.x, ob.y, ob.z)) +
                                             bnd.w - ob.w;
                                    }
                                    tighten(ub);
                                    rc = LC.w + m;
                                }
                                if (lane < cn) {
                                    const float4 ob = tab[o_os + c0 + lane];
                                    const float d2 = dist2(bnd.x, bnd.y, bnd.z, ob.x, ob.y, ob.z);
                                    h = within(d2, bnd.w + ob.w + m);
                                }
                                cand = __ballot_sync(kFull, h);
                                unsigned cm = cand;
                                while (cm) {
                                    const int o = __ffs(cm) - 1;
                                    cm &= cm - 1;
                                    const float4 ob = tab[o_os + c0 + o];
                                    const float d2 = dist2(cc.x, cc.y, cc.z, ob.x, ob.y, ob.z);
                                    own |= within(d2, rc + ob.w) ? (1u << o) : 0u;
                                }
                                if (MODE == kCount) {
                                    if (lane == 0) cnt[8] += cn;
                                    if (active) cnt[2] += __popc(cand);
                                }
                            }
                            if (cand == 0u) continue;  // nothing near
                            vote = true;
                            if (ra) {
                                hit |= fine_reassigned<false>(own, c0, ns, sf, F, m, tab, t, fr,
                                                              lane);
                                continue;
                            }
                            const unsigned wm = __reduce_or_sync(kFull, own);
                            if (MODE == kCount && active) {
                                cnt[4] += (unsigned long long)__popc(own) * ns;
                                own_any |= own != 0;
                            }
                            // fine stage: each of the link's spheres is placed once and
                            // tested against every obstacle of the warp's union mask
                            for (int s = 0; wm && s < ns; ++s) {
                                const float4 sp = tab[o_sph + sf + s];
                                const float3 p = apply(F, sp.x, sp.y, sp.z);
                                unsigned mm = wm;
                                while (mm) {
                                    const int o = __ffs(mm) - 1;
                                    mm &= mm - 1;
                                    const float4 ob = tab[o_os + c0 + o];
                                    const float d2 = dist2(p.x, p.y, p.z, ob.x, ob.y, ob.z);
                                    if (MODE == kClearance) {
                                        minc = fminf(minc, __fsqrt_rn(d2) - sp.w - ob.w);
                                    } else {
                                        const float th2 = sp.w + ob.w + m;
                                        hit |= d2 < th2 * th2;
                                    }
                                }
                            }
                        }

                        // ---- robot vs obstacle cuboids (oriented boxes); the tile and
                        // checkpoint levels test their bounding spheres against the box
                        // itself (distance to a convex set is 1-Lipschitz, so a sphere
                        // that encloses the fine spheres stays conservative)
                        for (int c0 = 0; c0 < NC; c0 += 32) {
                            const int cn = min(32, NC - c0);
                            unsigned own = 0, cand = 0;
                            {
                                if (MODE == kClearance) {
                                    // (no point of the box is farther than its
                                    // bounding sphere's far side)
                                    float ub = FLT_MAX;
                                    if (lane < cn) {
                                        const float4 cb0 = tab[o_oc + kCuboidF4 * (c0 + lane)];
                                        ub = __fsqrt_rn(dist2(bnd.x, bnd.y, bnd.z, cb0.x, cb0.y, cb0.z)) +
                                             bnd.w;
                                    }
                                    tighten(ub);
                                    rc = LC.w + m;
                                }
                                // the box's bounding sphere first (the box lies within
                                // it), its exact distance only when the sphere is near
                                bool h = false, exact = false;
                                if (lane < cn) {
                                    const float4 *cbp = tab + o_oc + kCuboidF4 * (c0 + lane);
                                    const float4 cb0 = cbp[0];
                                    const float dc2 = dist2(bnd.x, bnd.y, bnd.z, cb0.x, cb0.y, cb0.z);
                                    const float reach = cb0.w + bnd.w + m;
                                    exact = within(dc2, reach);
                                    if (exact) {
                                        const float d2 = box_dist2(bnd.x, bnd.y, bnd.z, cb0, cbp[1],
                                                                   cbp[2], cbp[3], cbp[4]);
                                        h = within(d2, bnd.w + m);
                                    }
                                }
                                cand = __ballot_sync(kFull, h);
                                unsigned cm = cand;
                                while (cm) {
                                    const int o = __ffs(cm) - 1;
                                    cm &= cm - 1;
                                    const float4 *cbp = tab + o_oc + kCuboidF4 * (c0 + o);
                                    const float d2 = box_dist2(cc.x, cc.y, cc.z, cbp[0], cbp[1],
                                                               cbp[2], cbp[3], cbp[4]);
                                    own |= within(d2, rc) ? (1u << o) : 0u;
                                }
                                if (MODE == kCount) {
                                    if (lane == 0) cnt[8] += cn;  // the bounding-sphere tests
                                    if (exact) cnt[11] += 1;
                                    if (active) cnt[10] += __popc(cand);
                                }
                            }
                            if (cand == 0u) continue;  // nothing near
                            vote = true;
                            if (ra) {
                                hit |= fine_reassigned<true>(own, c0, ns, sf, F, m, tab, t, fr,
                                                             lane);
                                continue;
                            }
                            const unsigned wm = __reduce_or_sync(kFull, own);
                            if (MODE == kCount && active) {
                                cnt[5] += (unsigned long long)__popc(own) * ns;
                                own_any |= own != 0;
                            }
                            for (int s = 0; wm && s < ns; ++s) {
                                const float4 sp = tab[o_sph + sf + s];
                                const float3 p = apply(F, sp.x, sp.y, sp.z);
                                unsigned mm = wm;
                                while (mm) {
                                    const int o = __ffs(mm) - 1;
                                    mm &= mm - 1;
                                    const float4 *cbp = tab + o_oc + kCuboidF4 * (c0 + o);
                                    const float d2 = box_dist2(p.x, p.y, p.z, cbp[0], cbp[1], cbp[2],
                                                               cbp[3], cbp[4]);
                                    if (MODE == kClearance) {
                                        minc = fminf(minc, __fsqrt_rn(d2) - sp.w);
                                    } else {
                                        const float th2 = sp.w + m;
                                        hit |= d2 < th2 * th2;
                                    }
                                }
                            }
                        }

                        // ---- robot vs earlier robots (links 0 .. l0-1) and, with
                        // self-collision, vs the links of this robot that its
                        // adjacency mask pairs with link l (bit i: link l0 + i)
                        const unsigned long long pm =
                            (l0 > 0 ? ~0ull >> (64 - l0) : 0ull) |
                            ((unsigned long long)(unsigned)__float_as_int(LB.w) << l0);
                        const unsigned pm0 = (unsigned)pm, pm1 = (unsigned)(pm >> 32);
                        if (pm) {
                            unsigned own0 = 0, own1 = 0, candp = 0;
                            {
                                if (MODE == kClearance) {
                                    float ub = FLT_MAX;
                                    if ((pm0 >> lane) & 1u) {
                                        const float4 o = tb[lane];
                                        ub = __fsqrt_rn(dist2(bnd.x, bnd.y, bnd.z, o.x, o.y, o.z)) + bnd.w +
                                             o.w;
                                        // (a link without spheres has no pair)
                                        if (__float_as_int(tab[o_link + kLinkF4 * lane + 1].z) == 0)
                                            ub = FLT_MAX;
                                    }
                                    tighten(ub);
                                }
                                // tile-level candidates: lane i tests link i (and i + 32)
                                bool h0 = false, h1 = false;
                                if ((pm0 >> lane) & 1u) {
                                    const float4 o = tb[lane];
                                    const float d2 = dist2(bnd.x, bnd.y, bnd.z, o.x, o.y, o.z);
                                    h0 = within(d2, bnd.w + o.w + m);
                                }
                                if ((pm1 >> lane) & 1u) {
                                    const float4 o = tb[lane + 32];
                                    const float d2 = dist2(bnd.x, bnd.y, bnd.z, o.x, o.y, o.z);
                                    h1 = within(d2, bnd.w + o.w + m);
                                }
                                const unsigned cand0 = __ballot_sync(kFull, h0);
                                const unsigned cand1 = __ballot_sync(kFull, h1);
                                for (int w = 0; w < 2; ++w) {
                                    unsigned cm = w == 0 ? cand0 : cand1;
                                    unsigned own = 0;
                                    while (cm) {
                                        const int bit = __ffs(cm) - 1;
                                        cm &= cm - 1;
                                        const int i = bit + 32 * w;
                                        const float4 LCi = tab[o_link + kLinkF4 * i + 2];
                                        const float *x = xc + (size_t)i * kXcFloats * 32 + lane;
                                        const float d2 = dist2(cc.x, cc.y, cc.z, x[0], x[32], x[64]);
                                        own |= within(d2, LC.w + LCi.w + m) ? (1u << bit) : 0u;
                                    }
                                    if (w == 0)
                                        own0 = own;
                                    else
                                        own1 = own;
                                }
                                if (MODE == kCount) {
                                    if (lane == 0) cnt[8] += __popcll(pm);
                                    if (active) cnt[3] += __popc(cand0) + __popc(cand1);
                                }
                                candp = cand0 | cand1;
                            }
                            if (candp != 0u) {
                            vote = true;
                            const unsigned w0 = __reduce_or_sync(kFull, own0);
                            const unsigned w1 = __reduce_or_sync(kFull, own1);
                            if (MODE == kCount && active) {
                                own_any |= (own0 | own1) != 0;
                                for (int w = 0; w < 2; ++w) {
                                    unsigned mm = w == 0 ? own0 : own1;
                                    while (mm) {
                                        const int i = __ffs(mm) - 1 + 32 * w;
                                        mm &= mm - 1;
                                        const int nsi =
                                            __float_as_int(tab[o_link + kLinkF4 * i + 1].z);
                                        cnt[6] += (unsigned long long)nsi * ns;
                                        cnt[7] += nsi;
                                    }
                                }
                            }
                            for (int w = 0; w < 2; ++w) {
                                unsigned mm = w == 0 ? w0 : w1;
                                while (mm) {
                                    const int i = __ffs(mm) - 1 + 32 * w;
                                    mm &= mm - 1;
                                    const Frame Fi = link_frame(tab, t, qa_s, dq_s, i, tk);
                                    const float4 LBi = tab[o_link + kLinkF4 * i + 1];
                                    const int sfi = __float_as_int(LBi.y), nsi = __float_as_int(LBi.z);
                                    // the other link's spheres four at a time, this
                                    // link's placed once per group of four
                                    for (int g0 = 0; g0 < nsi; g0 += 4) {
                                        float4 pa[4];
#pragma unroll
                                        for (int j = 0; j < 4; ++j) {
                                            const float4 sp2 = tab[o_sph + sfi + min(g0 + j, nsi - 1)];
                                            const float3 q3 = apply(Fi, sp2.x, sp2.y, sp2.z);
                                            pa[j] = make_float4(q3.x, q3.y, q3.z, sp2.w);
                                        }
                                        const int gn = min(4, nsi - g0);
                                        for (int s = 0; s < ns; ++s) {
                                            const float4 sp = tab[o_sph + sf + s];
                                            const float3 p = apply(F, sp.x, sp.y, sp.z);
#pragma unroll
                                            for (int j = 0; j < 4; ++j) {
                                                if (j >= gn) break;
                                                const float d2 =
                                                    dist2(p.x, p.y, p.z, pa[j].x, pa[j].y, pa[j].z);
                                                if (MODE == kClearance) {
                                                    minc = fminf(minc,
                                                                 __fsqrt_rn(d2) - sp.w - pa[j].w);
                                                } else {
                                                    const float th2 = sp.w + pa[j].w + m;
                                                    hit |= d2 < th2 * th2;
                                                }
                                            }
                                        }
                                    }
                                }
                            }
                            }  // candidates near link l
                        }
                        if (MODE == kCount && active && own_any) cnt[7] += ns;
                    }
                    if (MODE == kClearance && vote) tighten(FLT_MAX);
                    Tm = advance(F, LA.x, LA.y, LA.z, LA.w);
                    // a hit can only come from a fine stage of this link
                    if (MODE != kClearance && vote && __any_sync(kFull, hit)) goto tile_done;
                }
            }
        tile_done:
            if (MODE != kClearance && __any_sync(kFull, hit)) {
                edge_hit = true;
                break;
            }
        }

        if (MODE == kClearance) {
#pragma unroll
            for (int off = 16; off > 0; off >>= 1)
                minc = fminf(minc, __shfl_xor_sync(kFull, minc, off));
            if (lane == 0) P.min_clear[e] = minc;
        } else if (MODE == kVerdict) {
            if (lane == 0) {
                P.valid[e] = edge_hit ? 0 : 1;
                if (P.length) P.length[e] = len;
                if (P.npoints) P.npoints[e] = n;
            }
        }
    }

    if (MODE == kCount) {
#pragma unroll
        for (int c = 0; c < kCounters; ++c) {
            unsigned long long v = cnt[c];
#pragma unroll
            for (int off = 16; off > 0; off >>= 1) v += __shfl_xor_sync(kFull, v, off);
            if (lane == 0 && v) atomicAdd(P.counters + c, v);
        }
    }
    // The last warp to leave resets the work counter for the next launch on
    // this problem (every warp has made its final fetch before counting out).
    if (lane == 0) {
        __threadfence();
        if (atomicAdd(&P.work[1], 1) == P.total_warps - 1) {
            atomicExch(&P.work[0], 0);
            atomicExch(&P.work[1], 0);
        }
    }
}

// The same frame and interval count from (q_a, q_b - q_a) pairs.
__device__ __forceinline__ Frame link_frame(const float4 *tab, const Tables &t, const float2 *ad,
                                            int i, float tk) {
    int b = 0;
    while (t.link0[b + 1] <= i) ++b;
    Frame Tm = load_base(tab, t, b);
    for (int l = t.link0[b];; ++l) {
        const float4 LA = tab[t.off_link + kLinkF4 * l];
        float sn, cs;
        joint_sincos(__fmaf_rn(tk, ad[l].y, ad[l].x) + tab[t.off_link + kLinkF4 * l + 1].x, &sn, &cs);
        const Frame F = rotz(Tm, cs, sn);
        if (l == i) return F;
        Tm = advance(F, LA.x, LA.y, LA.z, LA.w);
    }
}

__device__ __forceinline__ int interval_count(const float2 *ad, int D, float res, float *len_out) {
    float acc = 0.f;
    for (int i = 0; i < D; ++i) acc = __fmaf_rn(ad[i].y, ad[i].y, acc);
    const float len = __fsqrt_rn(acc);
    const float nf = ceilf(__fdiv_rn(len, res));
    *len_out = len;
    if (!(nf >= 1.f)) return 1;
    return nf > 1073741824.f ? 1073741824 : (int)nf;
}

// A stored 16-bit grid coordinate as a float of kFieldMagic's scheme: differences
// of two are whole steps, exactly.  Each is within half a step of its
// coordinate, so a distance of two points in steps is within sqrt(3) of the
// true one: kGridSlack.
__device__ __forceinline__ float grid_float(unsigned v) {
    return __uint_as_float((unsigned)kFieldMagicBits + v);
}
constexpr float kGridSlack = 2.f;

// Fine robot-robot test of link l (frame F) against link i: true where a
// sphere of one touches a sphere of the other at the lane's checkpoint.  Only
// lanes whose own coarse spheres touch (own) can; each sphere of l is first
// tested against i's coarse sphere (grid coordinates x; it encloses i's spheres
// with slack), and i's spheres are placed when one of them is near.
__device__ __forceinline__ bool fine_pair(const float4 *tab, const Tables &t, const float2 *ad,
                                          float tk, const Frame &F, int l, int i,
                                          bool own, const uint16_t *x, float m) {
    const float4 LBl = tab[t.off_link + kLinkF4 * l + 1], LBi = tab[t.off_link + kLinkF4 * i + 1];
    const int sf = __float_as_int(LBl.y), ns = __float_as_int(LBl.z);
    const int sfi = __float_as_int(LBi.y), nsi = __float_as_int(LBi.z);
    const float pq = t.pq, pcx = t.pc[0], pcy = t.pc[1], pcz = t.pc[2];
    const float rci = tab[t.off_link + kLinkF4 * i + 2].w + m;
    const float xi = grid_float(x[0]), yi = grid_float(x[32]), zi = grid_float(x[64]);
    unsigned near = 0;  // spheres of l near i's coarse sphere in some lane
    for (int s = 0; s < ns; ++s) {
        const float4 sp = tab[t.off_sph + sf + s];
        const float3 p = apply(F, sp.x, sp.y, sp.z);
        const float th = fmaf(sp.w + rci, pq, kGridSlack);
        near |= own && dist2(fmaf(p.x, pq, pcx), fmaf(p.y, pq, pcy), fmaf(p.z, pq, pcz), xi, yi, zi) <
                           th * th
                    ? 1u << s : 0u;
    }
    near = __reduce_or_sync(kFull, near);
    if (!near) return false;
    const Frame Fi = link_frame(tab, t, ad, i, tk);
    bool hit = false;
    // i's spheres four at a time, each near sphere of l placed once per four
    for (int g0 = 0; g0 < nsi; g0 += 4) {
        float4 pa[4];
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            const float4 sp2 = tab[t.off_sph + sfi + min(g0 + j, nsi - 1)];
            const float3 q3 = apply(Fi, sp2.x, sp2.y, sp2.z);
            pa[j] = make_float4(q3.x, q3.y, q3.z, sp2.w);
        }
        for (unsigned mm = near; mm; mm &= mm - 1) {
            const float4 sp = tab[t.off_sph + sf + __ffs(mm) - 1];
            const float3 p = apply(F, sp.x, sp.y, sp.z);
#pragma unroll
            for (int j = 0; j < 4; ++j) {  // (a repeated last sphere changes nothing)
                const float d2 = dist2(p.x, p.y, p.z, pa[j].x, pa[j].y, pa[j].z);
                const float th2 = sp.w + pa[j].w + m;
                hit |= d2 < th2 * th2;
            }
        }
    }
    return hit;
}

// Link l against the links first + bit of mask (an earlier robot's, or its own
// robot's partners); near: lanes that may be in contact.  Coarse spheres at the
// lane's checkpoint, then the spheres of the pairs that some lane hit.
__device__ __forceinline__ bool link_pairs(const float4 *tab, const Tables &t, const float2 *ad,
                                           float tk, int l, bool near, int first,
                                           unsigned mask, const uint16_t *xc, float m) {
    const int lane = threadIdx.x & 31, o_link = t.off_link;
    const uint16_t *x = xc + l * (kXcFloats * 32) + lane;
    const float cx = grid_float(x[0]), cy = grid_float(x[32]), cz = grid_float(x[64]);
    const float rl = tab[o_link + kLinkF4 * l + 2].w + m, pq = t.pq;
    unsigned own = 0;
    for (unsigned mm = mask; mm; mm &= mm - 1) {
        const int bit = __ffs(mm) - 1, i = first + bit;
        if (__float_as_int(tab[o_link + kLinkF4 * i + 1].z) == 0) continue;  // no spheres
        const uint16_t *y = xc + i * (kXcFloats * 32) + lane;
        const float th = fmaf(rl + tab[o_link + kLinkF4 * i + 2].w, pq, kGridSlack);
        own |= near && dist2(cx, cy, cz, grid_float(y[0]), grid_float(y[32]), grid_float(y[64])) <
                           th * th
                   ? 1u << bit : 0u;
    }
    unsigned wi = __reduce_or_sync(kFull, own);
    if (!wi) return false;
    const Frame F = link_frame(tab, t, ad, l, tk);
    bool hit = false;
    for (; wi; wi &= wi - 1) {
        const int bit = __ffs(wi) - 1, i = first + bit;
        hit |= fine_pair(tab, t, ad, tk, F, l, i, (own >> bit) & 1u,
                         xc + i * (kXcFloats * 32) + lane, m);
    }
    return hit;
}

// Link l (its frame F and coarse centre cc at the lane's checkpoint) against
// the obstacles; near: lanes whose coarse sphere the distance field does not
// clear.  Tile bound over those lanes, lane-parallel obstacle tests, candidates
// against each lane's own coarse sphere, and the warp-wide union of what is hit
// against the link's fine spheres.
__device__ __forceinline__ bool link_obstacles(const float4 *tab, const Tables &t,
                                               const float4 &LB, const float4 &LC, const Frame &F,
                                               const float3 &cc, bool near, float m) {
    const int lane = threadIdx.x & 31;
    const int sf = __float_as_int(LB.y), ns = __float_as_int(LB.z);
    // one sphere around the near lanes' coarse spheres, from the box of their
    // centres taken relative to the workspace corner (coordinates >= 0, whose
    // bits order like unsigned integers)
    const float wlx = t.ws_lo[0], wly = t.ws_lo[1], wlz = t.ws_lo[2];
    const unsigned ux = __float_as_uint(cc.x - wlx), uy = __float_as_uint(cc.y - wly),
                   uz = __float_as_uint(cc.z - wlz);
    const float x0 = __uint_as_float(__reduce_min_sync(kFull, near ? ux : kFull));
    const float x1 = __uint_as_float(__reduce_max_sync(kFull, near ? ux : 0u));
    const float y0 = __uint_as_float(__reduce_min_sync(kFull, near ? uy : kFull));
    const float y1 = __uint_as_float(__reduce_max_sync(kFull, near ? uy : 0u));
    const float z0 = __uint_as_float(__reduce_min_sync(kFull, near ? uz : kFull));
    const float z1 = __uint_as_float(__reduce_max_sync(kFull, near ? uz : 0u));
    const float ex = 0.5f * (x1 - x0), ey = 0.5f * (y1 - y0), ez = 0.5f * (z1 - z0);
    float4 bnd;
    bnd.x = wlx + 0.5f * (x0 + x1);
    bnd.y = wly + 0.5f * (y0 + y1);
    bnd.z = wlz + 0.5f * (z0 + z1);
    // the hardware's approximate square root (an error of a few ulps), padded
    // by 2^-16 relative; kTileSlack covers the rest
    float rbox;
    asm("sqrt.approx.f32 %0, %1;" : "=f"(rbox) : "f"(fmaf(ex, ex, fmaf(ey, ey, ez * ez))));
    bnd.w = fmaf(rbox, 1.0000153f, LC.w + kTileSlack);
    if (!(bnd.w < FLT_MAX)) bnd.w = FLT_MAX * 2.f;  // never for finite inputs
    const float rc = LC.w + m;
    const int NS = t.NS, NC = t.NC;
    bool hit = false;
    for (int c0 = 0; c0 < NS; c0 += 32) {
        bool h = false;
        if (lane < NS - c0) {
            const float4 ob = tab[t.off_os + c0 + lane];
            const float th2 = bnd.w + ob.w + m;
            h = dist2(bnd.x, bnd.y, bnd.z, ob.x, ob.y, ob.z) < th2 * th2;
        }
        unsigned own = 0;
        for (unsigned cm = __ballot_sync(kFull, h); cm; cm &= cm - 1) {
            const int o = __ffs(cm) - 1;
            const float4 ob = tab[t.off_os + c0 + o];
            const float th2 = rc + ob.w;
            own |= near && dist2(cc.x, cc.y, cc.z, ob.x, ob.y, ob.z) < th2 * th2 ? 1u << o : 0u;
        }
        const unsigned wm = __reduce_or_sync(kFull, own);
        if (!wm) continue;
        // each of the link's spheres is placed once and tested against every
        // obstacle of the warp's union mask
        for (int s = 0; s < ns; ++s) {
            const float4 sp = tab[t.off_sph + sf + s];
            const float3 p = apply(F, sp.x, sp.y, sp.z);
            for (unsigned mm = wm; mm; mm &= mm - 1) {
                const float4 ob = tab[t.off_os + c0 + __ffs(mm) - 1];
                const float th2 = sp.w + ob.w + m;
                hit |= dist2(p.x, p.y, p.z, ob.x, ob.y, ob.z) < th2 * th2;
            }
        }
    }
    // cuboids: the bound against the box's bounding sphere (the box lies within
    // it), then its exact distance only where that sphere is near
    for (int c0 = 0; c0 < NC; c0 += 32) {
        bool h = false;
        if (lane < NC - c0) {
            const float4 *cbp = tab + t.off_oc + kCuboidF4 * (c0 + lane);
            const float4 cb0 = cbp[0];
            const float reach = cb0.w + bnd.w + m;
            if (dist2(bnd.x, bnd.y, bnd.z, cb0.x, cb0.y, cb0.z) < reach * reach) {
                const float th2 = bnd.w + m;
                h = box_dist2(bnd.x, bnd.y, bnd.z, cb0, cbp[1], cbp[2], cbp[3], cbp[4]) < th2 * th2;
            }
        }
        unsigned own = 0;
        for (unsigned cm = __ballot_sync(kFull, h); cm; cm &= cm - 1) {
            const int o = __ffs(cm) - 1;
            const float4 *cbp = tab + t.off_oc + kCuboidF4 * (c0 + o);
            own |= near && box_dist2(cc.x, cc.y, cc.z, cbp[0], cbp[1], cbp[2], cbp[3], cbp[4]) <
                               rc * rc
                       ? 1u << o : 0u;
        }
        const unsigned wm = __reduce_or_sync(kFull, own);
        if (!wm) continue;
        for (int s = 0; s < ns; ++s) {
            const float4 sp = tab[t.off_sph + sf + s];
            const float3 p = apply(F, sp.x, sp.y, sp.z);
            const float th2 = sp.w + m;
            for (unsigned mm = wm; mm; mm &= mm - 1) {
                const float4 *cbp = tab + t.off_oc + kCuboidF4 * (c0 + __ffs(mm) - 1);
                hit |= box_dist2(p.x, p.y, p.z, cbp[0], cbp[1], cbp[2], cbp[3], cbp[4]) < th2 * th2;
            }
        }
    }
    return hit;
}

// Verdicts of composite edges, one warp per edge and a checkpoint per lane.
// Per tile of 32 checkpoints and robot:
//   1. down the chain: forward kinematics in registers, the link's coarse
//      centre to shared memory, and one byte of the obstacles' distance field
//      at that centre, whose load overlaps the next link's frame and joint;
//   2. a link that the field does not clear in some lane runs the obstacle
//      tests (link_obstacles); a fine hit ends the edge;
//   3. robots in reach of each other (boxes around the tile's coarse centres,
//      one lane per earlier robot) run the link-pair tests: each link against
//      the earlier robot's box at the lane's own checkpoint, then against its
//      links, then sphere against sphere (fine_pair).
// Every level encloses what it replaces with a slack above FP32 rounding, and
// the sphere-level arithmetic alone decides.  Before, every link built a tile
// bound (six warp reductions) and tested it against all obstacles and earlier
// links, about 230 of the 279 instructions a link took; an eighth of the links
// now needs any of that (65,536 candidate edges of the table pair: 312 M
// instructions and 324 us before, 204 M and 237 us now; 8 arms, 4,099 edges:
// 57 M and 480 us, 32 M and 176 us).  Running all of a robot's links first and
// rebuilding the near ones' frames afterwards was slower (292 us: more joints
// before a colliding link ends the edge).
//
// SHARE: a warp that finds no edge left takes tiles of the edges that the block's
// other warps still work on: an edge's tiles are claimed one by one from its
// owner's words in shared memory, the first hit writes the verdict 0 and the
// warp that completes the last tile without one writes 1, so nobody waits.
// Without it a launch or a planner chunk ends with its longest edges, one warp
// each (8 arms, 4,099 edges: 256 us, with it 176).
//
// LOCAL: the edges [e0, e1) are handed out to the block's warps through the
// shared-memory counter *s_next (zeroed by the caller before the call) instead
// of the problem's global work counter, which is then left untouched.
//
// GROUP: the block's warps share one edge (edge blockIdx.x), tile after tile in
// turn, for batches of so few edges that an edge per warp would leave most of
// the chip idle: the time is then that of the longest edge, one tile after
// another.  The caller gives a shared flag (zero) in s_next.  With LOCAL too, the
// warps of each of the edges [e0, e1) are (P.warps / their number) in a row, s_next
// holds a zero flag for each, and the caller turns the flags into verdicts.
struct EdgeWords {
    // the owner's edge count (high half) and the next tile to claim (low half),
    // kClosed while the words below and the owner's joints are being written:
    // a claim is a compare-and-swap, so it only succeeds on the edge whose
    // words were read under the same count
    unsigned claim;
    int e, n;   // the edge and its interval count
    int T;      // its tiles
    int done;   // tiles completed without a hit
    int hit;
    int pad[2];
};
constexpr unsigned kClosed = 0xffffu;  // above any tile (32,769 at most)

template <bool LOCAL, bool GROUP = false, bool SHARE = !GROUP>
__device__ __forceinline__ void verdict_body(const VParams &P, float4 *sm4, int e0 = 0, int e1 = 0,
                                             int *s_next = nullptr) {
    float4 *tab = sm4;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const Tables &t = P.t;
    const int K = t.K, D = t.L;
    float *ws_all = reinterpret_cast<float *>(sm4 + t.n_f4);
    float *ws = ws_all + (size_t)warp * P.warp_floats + 8;
    float2 *ad = reinterpret_cast<float2 *>(ws);  // (q_a, q_b - q_a) of each joint, one spare
    auto words = [&](int w) {
        return reinterpret_cast<EdgeWords *>(ws_all + (size_t)w * P.warp_floats);
    };
    const int dpad = (D + 4) & ~3;                             // verdict_dpad
    int4 *rb = reinterpret_cast<int4 *>(ws + 2 * dpad);        // robot tile boxes [K][2]
    // coarse centres in grid coordinates [L][3][32]
    uint16_t *xc = reinterpret_cast<uint16_t *>(ws + 2 * dpad + 8 * K);

    for (int i = threadIdx.x; i < t.n_f4; i += blockDim.x) tab[i] = P.blob[i];
    if (SHARE && lane == 0 && warp < P.warps) words(warp)->claim = kClosed;
    __syncthreads();
    if (warp >= P.warps) return;  // spare warps of a shared multi-problem launch

    const int o_link = t.off_link;
    const uint8_t *df = t.df;
    const float fi = t.df_inv, fx = t.df_c[0], fy = t.df_c[1], fz = t.df_c[2];
    const unsigned fnx = t.df_n[0], fny = t.df_n[1], fnz = t.df_n[2];
    const int fout = t.df_out;
    const float pq = t.pq, pcx = t.pc[0], pcy = t.pc[1], pcz = t.pc[2];
    const float m = P.margin;
    if (lane == 0) ad[D] = make_float2(0.f, 0.f);
    const bool pairs = K > 1 || t.selfcol;
    const int split = GROUP ? (LOCAL ? P.warps / max(e1 - e0, 1) : P.warps) : 1;  // warps per edge
    int helping = 0;  // other warps looked at since the last edge (0: owner)
    for (;;) {
        int e = 0, n = 0, T = 0;
        bool edge_hit = false;
        EdgeWords *ew = words(warp);
        unsigned seen = 0;  // a helper's view of the owner's claim word
        if (!SHARE || helping == 0) {
            if (GROUP && LOCAL) {
                e = e0 + warp / split;
                if (e >= e1) return;
            } else if (GROUP) {
                e = blockIdx.x;
            } else {
                if (lane == 0) e = LOCAL ? e0 + atomicAdd(s_next, 1) : atomicAdd(&P.work[0], 1);
                e = __shfl_sync(kFull, e, 0);
                if (e >= (LOCAL ? e1 : P.E)) {
                    if (!SHARE) break;
                    helping = 1;
                    continue;
                }
            }
            if (SHARE && lane == 0) {
                const unsigned c = *(volatile unsigned *)&ew->claim;
                *(volatile unsigned *)&ew->claim = (c + 0x10000u) | kClosed;
                __threadfence_block();
            }
            __syncwarp();
            for (int i = lane; i < D; i += 32) {
                // (the persistent planner rewrites its edge buffers within one
                // launch: there the loads bypass the non-coherent cache)
                const float a =
                    LOCAL ? __ldcg(P.qa + (size_t)i * P.E + e) : __ldg(P.qa + (size_t)i * P.E + e);
                const float b =
                    LOCAL ? __ldcg(P.qb + (size_t)i * P.E + e) : __ldg(P.qb + (size_t)i * P.E + e);
                ad[i] = make_float2(a, __fsub_rn(b, a));
            }
            __syncwarp();
            float len;
            n = interval_count(ad, D, P.res, &len);
            // Edges beyond MRPOP_MAX_EDGE_INTERVALS intervals (or with non-finite
            // coordinates) are reported invalid without being checked.
            const bool too_long = !(len <= P.res * (float)MRPOP_MAX_EDGE_INTERVALS);
            T = too_long ? 0 : (n >> 5) + 1;  // ceil((n + 1) / 32)
            edge_hit = too_long;
            if (lane == 0 && (!GROUP || !LOCAL)) {
                if (P.length) P.length[e] = len;
                if (P.npoints) P.npoints[e] = n;
                if (SHARE && too_long) P.valid[e] = 0;
            }
            if (SHARE) {
                if (too_long) continue;
                if (T > 1 && lane == 0) {  // (a single tile is its owner's alone)
                    ew->e = e;
                    ew->n = n;
                    ew->T = T;
                    ew->done = ew->hit = 0;
                    __threadfence_block();
                    *(volatile unsigned *)&ew->claim &= ~0xffffu;  // open, tile 0 next
                }
                __syncwarp();
            }
        } else {
            // no edge is left to fetch: an owner's open edge is its last, which
            // it leaves only once every tile is claimed or one has hit
            if (helping >= P.warps) break;
            int w = warp + helping;
            if (w >= P.warps) w -= P.warps;
            ++helping;
            ew = words(w);
            int4 v = make_int4(0, 0, 0, 0);  // (one lane looks: the words may be changing)
            if (lane == 0) {
                const volatile EdgeWords *vw = ew;
                v.x = (int)vw->claim;
                __threadfence_block();
                v.y = vw->T;
                v.z = vw->e;
                v.w = vw->n;
                // closed, all claimed or hit: nothing to take
                if ((v.x & 0xffff) >= v.y || (v.x & 0xffff) == (int)kClosed || vw->hit) v.y = 0;
            }
            T = __shfl_sync(kFull, v.y, 0);
            if (T == 0) continue;
            seen = (unsigned)__shfl_sync(kFull, v.x, 0);
            e = __shfl_sync(kFull, v.z, 0);
            n = __shfl_sync(kFull, v.w, 0);
            const float2 *from = reinterpret_cast<const float2 *>(ew + 1);
            __syncwarp();
            for (int i = lane; i < D; i += 32) ad[i] = from[i];
            __syncwarp();
        }

        volatile int *flag = GROUP ? s_next + (LOCAL ? e - e0 : 0) : nullptr;
        for (int own = GROUP ? warp % split : 0;; own += split) {
            int tile = own;
            if (!SHARE) {
                if (tile >= T || edge_hit) break;
                // another warp's tile collides: one lane reads the flag, which that
                // warp may be writing, so that the whole warp leaves or stays
                if (GROUP && __shfl_sync(kFull, lane == 0 ? *flag : 0, 0)) break;
            } else if (T > 1) {
                if (lane == 0) {
                    tile = T;
                    if (!*(volatile int *)&ew->hit) {
                        if (helping == 0) {
                            tile = (int)(atomicAdd(&ew->claim, 1u) & 0xffffu);
                        } else {
                            __threadfence_block();
                            unsigned c = *(volatile unsigned *)&ew->claim;
                            while ((c >> 16) == (seen >> 16) && (int)(c & 0xffffu) < T) {
                                const unsigned got = atomicCAS(&ew->claim, c, c + 1u);
                                if (got == c) {
                                    tile = (int)(c & 0xffffu);
                                    break;
                                }
                                c = got;
                            }
                        }
                    }
                }
                tile = __shfl_sync(kFull, tile, 0);
                if (tile >= T) break;
                if (helping) helping = 1;  // look at every warp again afterwards
            }
            int k = P.order ? tile * 32 + lane : tile + T * lane;
            k = min(k, n);
            // (k = 0 apart: a zero numerator sends the whole warp through the
            // division's slow path)
            const float tq = __fdiv_rn((float)max(k, 1), (float)n);
            const float tk = k > 0 ? tq : 0.f;
            float sn, cs;  // of the next link's joint
            joint_sincos(__fmaf_rn(tk, ad[0].y, ad[0].x) + tab[o_link + 1].x, &sn, &cs);
            for (int b = 0; b < K && !edge_hit; ++b) {
                const int l0 = t.link0[b], l1 = t.link0[b + 1];
                Frame Tm = load_base(tab, t, b);
                // box of the lane's centres (float bits, positive: ordered)
                unsigned bx0 = kFull, by0 = kFull, bz0 = kFull, bx1 = 0, by1 = 0, bz1 = 0;
                const float4 *lk = tab + o_link + kLinkF4 * l0;
                uint16_t *x = xc + l0 * (kXcFloats * 32) + lane;
                const float2 *aj = ad + l0 + 1;  // the next link's joint
                const float rmax = lk[3].y;  // the robot's largest coarse radius, -1: no spheres
                bool hit = false;
#pragma unroll 1
                for (int l = l0; l < l1; ++l) {
                    const float4 LA = lk[0], LC = lk[2], LD = lk[3];
                    const Frame F = rotz(Tm, cs, sn);
                    const float3 cc = apply(F, LC.x, LC.y, LC.z);
                    // the field's byte, loaded ahead of the next link's frame and joint
                    const int th = __float_as_int(LD.x);
                    const unsigned ix = __float_as_uint(fmaf(cc.x, fi, fx)) - kFieldMagicBits;
                    const unsigned iy = __float_as_uint(fmaf(cc.y, fi, fy)) - kFieldMagicBits;
                    const unsigned iz = __float_as_uint(fmaf(cc.z, fi, fz)) - kFieldMagicBits;
                    const bool in = (ix < fnx) & (iy < fny) & (iz < fnz);
                    int v = fout;
                    if (in) v = __ldg(df + ((iz * fny + iy) * fnx + ix));
                    Tm = advance(F, LA.x, LA.y, LA.z, LA.w);
                    // (the last link's successor is the spare entry)
                    const float2 qd = *aj++;
                    joint_sincos(__fmaf_rn(tk, qd.y, qd.x) + LD.z, &sn, &cs);
                    if (pairs) {
                        const unsigned gx = __float_as_uint(fmaf(cc.x, pq, pcx));
                        const unsigned gy = __float_as_uint(fmaf(cc.y, pq, pcy));
                        const unsigned gz = __float_as_uint(fmaf(cc.z, pq, pcz));
                        x[0] = (uint16_t)gx;
                        x[32] = (uint16_t)gy;
                        x[64] = (uint16_t)gz;
                        // (a link without spheres only widens the box)
                        bx0 = min(bx0, gx);
                        bx1 = max(bx1, gx);
                        by0 = min(by0, gy);
                        by1 = max(by1, gy);
                        bz0 = min(bz0, gz);
                        bz1 = max(bz1, gz);
                    }
                    const bool near = v < th;
                    if (__any_sync(kFull, near)) {
                        hit = link_obstacles(tab, t, lk[1], LC, F, cc, near, m);
                        if (__any_sync(kFull, hit)) {
                            edge_hit = true;
                            break;
                        }
                    }
                    lk += kLinkF4;
                    x += kXcFloats * 32;
                }
                if (edge_hit || rmax < 0.f) {
                    if (lane == 0) rb[2 * b].w = __float_as_int(-1.f);  // no spheres: pairs with nothing
                    continue;
                }
                if (K > 1) {
                    // the robot's box over the tile
                    int4 lo, hi;
                    lo.x = (int)__reduce_min_sync(kFull, bx0);
                    hi.x = (int)__reduce_max_sync(kFull, bx1);
                    lo.y = (int)__reduce_min_sync(kFull, by0);
                    hi.y = (int)__reduce_max_sync(kFull, by1);
                    lo.z = (int)__reduce_min_sync(kFull, bz0);
                    hi.z = (int)__reduce_max_sync(kFull, bz1);
                    lo.w = __float_as_int(rmax);
                    hi.w = 0;
                    if (lane == 0) {
                        rb[2 * b] = lo;
                        rb[2 * b + 1] = hi;
                    }
                    __syncwarp();
                    bool close = false;
                    if (lane < b) {
                        const int4 ol = rb[2 * lane], oh = rb[2 * lane + 1];
                        const float gx = (float)max(max(ol.x - hi.x, lo.x - oh.x), 0);
                        const float gy = (float)max(max(ol.y - hi.y, lo.y - oh.y), 0);
                        const float gz = (float)max(max(ol.z - hi.z, lo.z - oh.z), 0);
                        const float ro = __int_as_float(ol.w);
                        const float r = fmaf(ro + rmax + m + kTileSlack, pq, kGridSlack);
                        close = ro >= 0.f && fmaf(gx, gx, fmaf(gy, gy, gz * gz)) < r * r;
                    }
                    for (unsigned cm = __ballot_sync(kFull, close); cm; cm &= cm - 1) {
                        const int a = __ffs(cm) - 1;
                        const int a0 = t.link0[a], a1 = t.link0[a + 1];
                        // robot a's box at the lane's checkpoint
                        unsigned ux0 = kFull, uy0 = kFull, uz0 = kFull, ux1 = 0, uy1 = 0, uz1 = 0;
                        for (int i = a0; i < a1; ++i) {
                            const uint16_t *x = xc + i * (kXcFloats * 32) + lane;
                            const unsigned vx = x[0], vy = x[32], vz = x[64];
                            ux0 = min(ux0, vx);
                            ux1 = max(ux1, vx);
                            uy0 = min(uy0, vy);
                            uy1 = max(uy1, vy);
                            uz0 = min(uz0, vz);
                            uz1 = max(uz1, vz);
                        }
                        const float ax0 = grid_float(ux0), ay0 = grid_float(uy0), az0 = grid_float(uz0);
                        const float ax1 = grid_float(ux1), ay1 = grid_float(uy1), az1 = grid_float(uz1);
                        const float ra = __int_as_float(rb[2 * a].w) + m + kTileSlack;
                        unsigned nl = 0;
                        for (int l = l0; l < l1; ++l) {
                            if (__float_as_int(tab[o_link + kLinkF4 * l + 3].x) == 0) continue;
                            const uint16_t *x = xc + l * (kXcFloats * 32) + lane;
                            const float vx = grid_float(x[0]), vy = grid_float(x[32]),
                                        vz = grid_float(x[64]);
                            const float gx = fmaxf(fmaxf(ax0 - vx, vx - ax1), 0.f);
                            const float gy = fmaxf(fmaxf(ay0 - vy, vy - ay1), 0.f);
                            const float gz = fmaxf(fmaxf(az0 - vz, vz - az1), 0.f);
                            const float r = fmaf(tab[o_link + kLinkF4 * l + 2].w + ra, pq, kGridSlack);
                            nl |= fmaf(gx, gx, fmaf(gy, gy, gz * gz)) < r * r ? 1u << (l - l0) : 0u;
                        }
                        for (unsigned wl = __reduce_or_sync(kFull, nl); wl; wl &= wl - 1) {
                            const int j = __ffs(wl) - 1;
                            const unsigned links = ((1u << (a1 - a0)) - 1u);
                            hit |= link_pairs(tab, t, ad, tk, l0 + j, (nl >> j) & 1u, a0,
                                              links, xc, m);
                            if (__any_sync(kFull, hit)) {
                                edge_hit = true;
                                break;
                            }
                        }
                        if (edge_hit) break;
                    }
                }
                if (t.selfcol && !edge_hit)
                    for (int l = l0; l < l1 && !edge_hit; ++l) {
                        const unsigned mask = __float_as_int(tab[o_link + kLinkF4 * l + 1].w);
                        if (!mask || __float_as_int(tab[o_link + kLinkF4 * l + 3].x) == 0) continue;
                        hit |= link_pairs(tab, t, ad, tk, l, true, l0, mask, xc, m);
                        edge_hit = __any_sync(kFull, hit);
                    }
            }
            if (SHARE) {
                if (lane == 0) {
                    if (T == 1) {
                        P.valid[e] = edge_hit ? 0 : 1;
                    } else if (edge_hit) {
                        *(volatile int *)&ew->hit = 1;
                        P.valid[e] = 0;
                    } else if (atomicAdd(&ew->done, 1) == T - 1) {
                        P.valid[e] = 1;
                    }
                }
                if (edge_hit || tile == T - 1) break;  // (every tile is claimed)
            }
        }
        if (GROUP) {
            if (lane == 0 && edge_hit) *flag = 1;
            if (LOCAL) return;
            __syncthreads();
            if (threadIdx.x == 0) P.valid[e] = *flag == 0;
            return;
        }
        if (!SHARE && lane == 0) P.valid[e] = edge_hit ? 0 : 1;
    }
    // The last warp to leave resets the work counter for the next launch on
    // this problem (every warp has made its final fetch before counting out).
    if (!LOCAL && lane == 0) {
        __threadfence();
        if (atomicAdd(&P.work[1], 1) == P.total_warps - 1) {
            atomicExch(&P.work[0], 0);
            atomicExch(&P.work[1], 0);
        }
    }
}

}  // namespace vb
}  // namespace mrpop
