// em_kernels.cu -- fused E-step / M-step statistics, reduction and FP64 finalize.
//
// GIRA (arXiv 2307.00071) Sec. V: the E-step of Eq. (estep) is evaluated in the
// log domain (Eq. logestep) with the Cholesky form of the log-density
// (Eq. simplifiedGaussian); the M-step (standard full-covariance update, not
// written in the paper) is fed by per-component sufficient statistics.
//
// estep_pt_kernel (K <= 1024, 3-D; point-stationary): a block of 128 points stays in
// the registers of two warps, which split the component pairs; every pair's parameters
// come from shared memory as broadcasts, two components per packed operation
// (FADD2/FMUL2/FFMA2).  Phase 1 takes e_nb = 2^(l_nb - cmax) and the per-point totals,
// phase 2 the per-component statistics S0 = sum r, S1 = sum r y, S2 = sum r y y^T with
// y = P'(x - mu_old), for the pairs that are live in the block.  The responsibility
// matrix is never stored.  A pair out of reach of the block's box is skipped: its e is
// exactly 0 for every point (ex2.approx.ftz returns +0 below 2^-126) and a zero term
// changes no sum.  Points and components run in Morton order, so most pairs are out of
// reach.  Larger K and 4-D: reach_kernels.cu; the gradient: adjoint_kernels.cu.
#include <cxxabi.h>
#include <float.h>
#include <math.h>

#include <algorithm>
#include <cstdlib>
#include <string>

#include "gira_internal.cuh"

namespace gira {

namespace {

constexpr unsigned FULL = 0xffffffffu;
constexpr float LN2F = 0.693147180559945309f;
constexpr double LN2 = 0.693147180559945309417232121458;

// Log-density in base 2 for a component pair and one point (pairs packed).
struct PairParams {
    float2 p[6], c, nmu[3], w;
};

// P.c holds (cmax - c) >= 0: q' = |y|^2 + (cmax - c), y = P'(x - mu), and the
// logit relative to cmax is -q'.  The difference x - mu is taken first: it is
// exact or nearly so for the points a component reaches, so y carries only a
// few roundings relative to itself.  (The expanded form P'x + b' with
// b' = -P'mu would cancel two numbers of size |P'||x| -- a point metres from
// the origin against a millimetre-thin component: ~10^3 -- and carry the
// binary32 rounding of b' into every y; measured on the frame, one EM
// iteration in that form moves weights and covariances 10-20 times further from
// the binary64 result than this one.)
__device__ __forceinline__ float2 neg_logit2(const PairParams& P, float2 X0, float2 X1, float2 X2) {
    const float2 d0 = add2(X0, P.nmu[0]), d1 = add2(X1, P.nmu[1]), d2 = add2(X2, P.nmu[2]);
    const float2 y0 = mul2(P.p[0], d0);
    const float2 y1 = fma2(P.p[2], d1, mul2(P.p[1], d0));
    const float2 y2 = fma2(P.p[5], d2, fma2(P.p[4], d1, mul2(P.p[3], d0)));
    return fma2(y2, y2, fma2(y1, y1, fma2(y0, y0, P.c)));
}

// The same, also returning the whitened coordinates y = P'(x - mu) it formed
// (the same operations, so the same bits).
__device__ __forceinline__ float2 neg_logit2_y(const PairParams& P, float2 X0, float2 X1, float2 X2, float2& y0,
                                               float2& y1, float2& y2) {
    const float2 d0 = add2(X0, P.nmu[0]), d1 = add2(X1, P.nmu[1]), d2 = add2(X2, P.nmu[2]);
    y0 = mul2(P.p[0], d0);
    y1 = fma2(P.p[2], d1, mul2(P.p[1], d0));
    y2 = fma2(P.p[5], d2, fma2(P.p[4], d1, mul2(P.p[3], d0)));
    return fma2(y2, y2, fma2(y1, y1, fma2(y0, y0, P.c)));
}

constexpr long long MBAR_POLL_LIMIT = 2000000000ll;   // bound on any mbarrier wait: 2 s of wall time

// ------------------------------------------------------------------ point-stationary E-step
// The E-step with the roles of the operands the other way round: each lane owns
// PT_P points in registers (a warp: 32 PT_P consecutive points), and every pair
// of components is read from shared memory as a broadcast (the CTA's copy of
// the parameters, staged once by one TMA bulk copy).  Per-point sums stay in
// their lane: no cross-lane or cross-warp reduction, no barrier.
//  phase 1  for every pair: both logits at the lane's points, e = 2^-q', the
//           per-point totals; one warp vote records whether the pair reaches any
//           point of the warp (some e nonzero: ex2.approx.ftz gives exact zeros);
//  totals   1 / total per point and the log-likelihood; a point whose total
//           falls below 2^-100 takes the exact per-point maximum (Eq. logestep's
//           max-subtraction) and makes every pair live for its warp;
//  phase 2  for the live pairs only: e again (the same instructions, so the same
//           bits), the statistics of both components over the warp's points in
//           whitened coordinates y = P'(x - mu_old) -- S0 = sum r, S1 = sum r y,
//           S2 = sum r y y^T -- reduced over the warp's lanes and written to the
//           warp's partials; the warp's live mask tells the finalize which ones.
// With the components in space-filling-curve order a warp's 128 neighbouring
// points reach about a sixth of the pairs (the depth frame at K = 512), and the
// other pairs cost only phase 1.  The statistics are sums of the same terms as
// the other kernels' in another order.
// Relative costs of a listed pair (phase 1) and a live pair (phase 2) per point,
// and the 8-bit logarithmic key of a CTA's work (16 steps per octave) by which
// the finalize orders the CTAs of a later iteration.
constexpr unsigned PT_COST_NEAR = 26, PT_COST_LIVE = 54;
__device__ __forceinline__ uint8_t work_key(unsigned w) {
    const int e = 31 - __clz(w | 1u);
    const unsigned m = (e >= 4 ? (w >> (e - 4)) : (w << (4 - e))) & 15u;
    return (uint8_t)min(255u, (unsigned)e * 16u + m);
}
constexpr int PT_P = 4;           // points per lane
constexpr int PT_W = 4;           // warps per CTA
constexpr int PT_H = 2;           // warps sharing a block of 32 * PT_P points (the pairs split between them)
constexpr int PT_B = PT_W / PT_H; // point blocks per CTA: partial rows and mask rows per CTA
constexpr int PT_PTS = 32 * PT_P * PT_B;   // points per CTA

// Pairs the kernel reads for k components: ceil(k / 2) rounded up to a multiple
// of 32 (never beyond the padded parameter block, whose extra slots are padding
// components with c = -inf).
__host__ __device__ constexpr int pt_pairs(int k) { return (((k + 1) / 2) + 31) & ~31; }
// floats of one partial row: [pairs][2 NSTAT], a pair's values 80 contiguous bytes
__host__ __device__ constexpr int pt_row_floats(int k) { return ((k + 1) / 2) * 2 * NSTAT; }
constexpr float PT_REACH = 128.f;  // q' above which a component is out of reach (e = 0 from q' > 126)
// parameters, then per warp the live-mask words and the list of reachable pairs
__host__ __device__ constexpr size_t pt_smem_bytes(int k) {
    return (size_t)pt_pairs(k) * PAIR_FLOATS * 4 + (size_t)PT_W * (pt_pairs(k) / 32) * 4 +
           (size_t)PT_W * pt_pairs(k) * 2;
}

// Sum of 20 values (10 float2: component 2p in .x, 2p+1 in .y) over the warp's
// lanes.  On return lane l with (l & 7) < 5 holds value 10 (l >> 4) + 5 ((l >> 3) & 1) + (l & 7):
// halving exchanges for the first two levels, butterflies for the last three.
__device__ __forceinline__ float pt_warp_reduce20(const float2 (&S)[NSTAT], int lane, int* vidx) {
    const bool b4 = lane & 16, b3 = lane & 8;
    float w[NSTAT];
#pragma unroll
    for (int i = 0; i < NSTAT; ++i) {
        const float keep = b4 ? S[i].y : S[i].x, send = b4 ? S[i].x : S[i].y;
        w[i] = keep + __shfl_xor_sync(FULL, send, 16);
    }
    float z[5];
#pragma unroll
    for (int i = 0; i < 5; ++i) {
        const float keep = b3 ? w[5 + i] : w[i], send = b3 ? w[i] : w[5 + i];
        z[i] = keep + __shfl_xor_sync(FULL, send, 8);
    }
#pragma unroll
    for (int o = 4; o > 0; o >>= 1)
#pragma unroll
        for (int i = 0; i < 5; ++i) z[i] += __shfl_xor_sync(FULL, z[i], o);
    const int i = lane & 7;
    *vidx = 10 * (b4 ? 1 : 0) + 5 * (b3 ? 1 : 0) + i;
    return i == 0 ? z[0] : i == 1 ? z[1] : i == 2 ? z[2] : i == 3 ? z[3] : z[4];
}

// The barrier of point block blk's PT_H warps (barrier ids known at compile time,
// so the kernel holds PT_B + 1 of them).
__device__ __forceinline__ void pt_block_sync(int blk) {
    static_assert(PT_B == 2 && PT_H == 2, "one named barrier per point block");
    if (blk == 0) asm volatile("bar.sync 1, %0;" ::"n"(32 * PT_H) : "memory");
    else asm volatile("bar.sync 2, %0;" ::"n"(32 * PT_H) : "memory");
}

template <bool STATS>
__global__ void __launch_bounds__(32 * PT_W, 4) estep_pt_kernel(const EStepLaunch a_in) {
    extern __shared__ __align__(128) unsigned char dsm[];
    __shared__ __align__(8) uint64_t bar_tma;
    __shared__ int s_skip, s_norm, s_dead;
    __shared__ double s_ll[PT_W];
    __shared__ unsigned s_pairs[PT_W][2];
    __shared__ float2 s_tot[PT_W][PT_P][32];   // phase-1 sums of every warp, for its partner
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int blk = warp / PT_H, half = warp % PT_H;   // point block; which pairs (pp % PT_H == half)
    int cta = blockIdx.x;
    // the instance's first point (batched launches); the loads below index the
    // launch's own pointer by it (loads through the pointer advanced in the local
    // copy of the launch struct read the unadvanced one under nvcc 13.0 for sm_103a)
    int64_t pt0 = 0;
    EStepLaunch a = a_in;
    if (a_in.units) {
        const BatchUnit u = a_in.units[blockIdx.x];
        const BatchInst I = a_in.insts[u.inst];
        cta = u.cta;
        pt0 = I.pt_off;
        a.n = I.n;
        a.k = I.k;
        a.params = a_in.params + I.par_off;
        a.partials = a_in.partials ? a_in.partials + I.part_off : nullptr;
        a.masks = a_in.masks ? a_in.masks + I.mask_off : nullptr;
        a.pt_rows = (int64_t)I.ctas * PT_B;
        a.ll_partials = a_in.ll_partials ? a_in.ll_partials + I.ll_off : nullptr;
        a.per_point = a_in.per_point ? a_in.per_point + I.pt_off : nullptr;
        a.st = a_in.states + u.inst;
    }
    if (a_in.cta_perm && a_in.iter >= 3) {   // the order the finalize chose two iterations ago
        const int c = a_in.cta_perm[(size_t)(a_in.iter & 1) * gridDim.x + blockIdx.x];
        if (GIRA_IN(c >= 0 && c < (int)gridDim.x, a.st)) cta = c;
    }
    // pairs evaluated: ceil(k / 2) rounded up to even (within the padded block, whose
    // extra slots are padding components with c = -inf); mask words for pt_pairs(k)
    const int npairs = ((((a.k + 1) >> 1) + 1) & ~1);
    const int nwords = pt_pairs(a.k) / 32;
    const float4* spar = reinterpret_cast<const float4*>(dsm);   // [npairs][PAIR_F4]
    uint32_t* smask_all = reinterpret_cast<uint32_t*>(dsm + (size_t)pt_pairs(a.k) * PAIR_FLOATS * 4);
    uint32_t* smask = smask_all + warp * nwords;   // [nwords] live bits of the warp's pairs
    uint16_t* slist = reinterpret_cast<uint16_t*>(smask_all + PT_W * nwords) + warp * pt_pairs(a.k);
    // the lane's points (never written inside a fit: loaded before the wait); a slot
    // beyond n holds a point 1e18 m away, where every q' is +inf and e exactly 0
    const int64_t base = (int64_t)cta * PT_PTS + (int64_t)blk * 32 * PT_P + lane;
    float2 X[PT_P][3];
    bool valid[PT_P];
#pragma unroll
    for (int p = 0; p < PT_P; ++p) {
        const int64_t i = base + 32 * p;
        valid[p] = i < a.n && GIRA_IN(a_in.n_buf == 0 || pt0 + i < a_in.n_buf, a.st);
        if (valid[p]) {
            const float4 xy = a_in.pts8[2 * (pt0 + i)], zz = a_in.pts8[2 * (pt0 + i) + 1];
            X[p][0] = f2(xy.x, xy.y);
            X[p][1] = f2(xy.z, xy.w);
            X[p][2] = f2(zz.x, zz.y);
        } else {
            X[p][0] = X[p][1] = X[p][2] = dup(1e18f);
        }
    }
    pdl_wait();   // the parameters and the state written by the previous kernel
    if (threadIdx.x == 0) {
        s_skip = (a.iter > a.st->stop_after) || (a.st->error != 0);
        s_norm = a.st->w_raw;
        s_dead = 0;
        if (!s_skip) {
            mbar_init(&bar_tma, 1);
            mbar_fence_init();
            const uint32_t bytes = (uint32_t)npairs * PAIR_FLOATS * 4u;
            mbar_expect_tx(&bar_tma, bytes);
            tma_load_1d(reinterpret_cast<void*>(dsm), a.params, bytes, &bar_tma);
            if (!mbar_wait_bounded(&bar_tma, 0u, MBAR_POLL_LIMIT)) {
                s_dead = 1;
                set_error(a.st, GIRA_ERR_TIMEOUT);
                mbar_wait_bounded(&bar_tma, 0u, MBAR_POLL_LIMIT);   // let the copy land
            }
        }
    }
    __syncthreads();
    if (s_skip || s_dead) return;
    pdl_allow_next();

    // reference cmax = max_b c_b and the weight normaliser (every warp, same order)
    float cm = -INFINITY, wsv = 0.f;
    for (int pp = lane; pp < npairs; pp += 32) {
        const float4 v4 = spar[pp * PAIR_F4 + 4], v6 = spar[pp * PAIR_F4 + 6];
        cm = fmaxf(cm, fmaxf(v4.z, v4.w));
        wsv += v6.z + v6.w;
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        cm = fmaxf(cm, __shfl_xor_sync(FULL, cm, o));
        wsv += __shfl_xor_sync(FULL, wsv, o);
    }
    const float cmax = cm;
    const float ref0 = s_norm ? cmax - __log2f(wsv) : cmax;

    auto load_pair = [&](int pp, PairParams& P) {
        if (!GIRA_IN(pp >= 0 && pp < npairs, a.st)) pp = 0;
        const float4* q = spar + (size_t)pp * PAIR_F4;
        const float4 v0 = q[0], v1 = q[1], v2 = q[2], v4 = q[4], v5 = q[5], v6 = q[6];
        P.p[0] = f2(v0.x, v0.y); P.p[1] = f2(v0.z, v0.w);
        P.p[2] = f2(v1.x, v1.y); P.p[3] = f2(v1.z, v1.w);
        P.p[4] = f2(v2.x, v2.y); P.p[5] = f2(v2.z, v2.w);
        P.c = f2(cmax - v4.z, cmax - v4.w);
        P.nmu[0] = f2(v5.x, v5.y); P.nmu[1] = f2(v5.z, v5.w);
        P.nmu[2] = f2(v6.x, v6.y);
    };

    // ---- phase 0: the pairs that can reach a point of the warp.  Over the box of
    // the warp's points, two lower bounds of q' = |P'(x - mu)|^2 + (cmax - c):
    //   |P'(x - mu)| >= |P'(ctr - mu)| - sum_j h_j |column j of P'|  (h: half-extents)
    //   |P'(x - mu)|^2 >= sigma_min(P')^2 dist(mu, box)^2
    // A component whose bound exceeds PT_REACH (with relative slack for the binary32
    // rounding of the bound and of q' itself) has q' > 126 at every point of the warp,
    // where ex2.approx.ftz gives exact zeros: skipping it leaves every sum unchanged.
    int nlive = 0;
    {
        float lo[3], hi[3];
#pragma unroll
        for (int j = 0; j < 3; ++j) {
            lo[j] = INFINITY;
            hi[j] = -INFINITY;
        }
#pragma unroll
        for (int p = 0; p < PT_P; ++p)
            if (valid[p])
#pragma unroll
                for (int j = 0; j < 3; ++j) {
                    lo[j] = fminf(lo[j], X[p][j].x);
                    hi[j] = fmaxf(hi[j], X[p][j].x);
                }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1)
#pragma unroll
            for (int j = 0; j < 3; ++j) {
                lo[j] = fminf(lo[j], __shfl_xor_sync(FULL, lo[j], o));
                hi[j] = fmaxf(hi[j], __shfl_xor_sync(FULL, hi[j], o));
            }
        const bool any_point = lo[0] <= hi[0];
        float ctr[3], h[3];
#pragma unroll
        for (int j = 0; j < 3; ++j) {
            ctr[j] = 0.5f * (lo[j] + hi[j]);
            h[j] = fmaxf(hi[j] - ctr[j], ctr[j] - lo[j]);
        }
        for (int j0 = 0; j0 < npairs; j0 += 32 * PT_H) {   // this warp's pairs: pp % PT_H == half
            const int pp = j0 + PT_H * lane + half;
            bool live = false;
            if (any_point && pp < npairs) {
                const float4* q = spar + (size_t)pp * PAIR_F4;
                const float4 v0 = q[0], v1 = q[1], v2 = q[2], v4 = q[4], v5 = q[5], v6 = q[6], v7 = q[7];
                const float pc[2][6] = {{v0.x, v0.z, v1.x, v1.z, v2.x, v2.z}, {v0.y, v0.w, v1.y, v1.w, v2.y, v2.w}};
                const float nm[2][3] = {{v5.x, v5.z, v6.x}, {v5.y, v5.w, v6.y}};
                const float cc[2] = {v4.z, v4.w}, s2[2] = {v7.x, v7.y};
#pragma unroll
                for (int m = 0; m < 2; ++m) {
                    const float room = PT_REACH - (cmax - cc[m]);   // q' budget left for |y|^2
                    const float* P = pc[m];
                    const float d0 = ctr[0] + nm[m][0], d1 = ctr[1] + nm[m][1], d2 = ctr[2] + nm[m][2];
                    const float y0 = P[0] * d0, y1 = fmaf(P[2], d1, P[1] * d0);
                    const float y2 = fmaf(P[5], d2, fmaf(P[4], d1, P[3] * d0));
                    const float yy = fmaf(y2, y2, fmaf(y1, y1, y0 * y0));
                    const float r = fmaf(h[0], sqrtf(fmaf(P[0], P[0], fmaf(P[1], P[1], P[3] * P[3]))),
                                         fmaf(h[1], sqrtf(fmaf(P[2], P[2], P[4] * P[4])), h[2] * fabsf(P[5])));
                    const float reach = (r + sqrtf(fmaxf(room, 0.f))) * (1.f + 1.f / 256.f);
                    const float e0 = fmaxf(fabsf(d0) - h[0], 0.f), e1 = fmaxf(fabsf(d1) - h[1], 0.f),
                                e2 = fmaxf(fabsf(d2) - h[2], 0.f);
                    const float iso = s2[m] * fmaf(e2, e2, fmaf(e1, e1, e0 * e0)) * (1.f - 1.f / 128.f);
                    live = live || (room > 0.f && yy <= reach * reach && iso <= room);
                }
            }
            const uint32_t m = __ballot_sync(FULL, live);
            const int at = nlive + __popc(m & ((1u << lane) - 1u));
            if (live && GIRA_IN(at < pt_pairs(a.k), a.st)) slist[at] = (uint16_t)pp;
            nlive += __popc(m);
        }
    }
    __syncwarp();

    // ---- phase 1: the reachable pairs, the lane's points (two pairs per step)
    if (STATS && lane < nwords) smask[lane] = 0u;
    __syncwarp();
    float2 tot[PT_P];
#pragma unroll
    for (int p = 0; p < PT_P; ++p) tot[p] = f2(0.f, 0.f);
    for (int i = 0; i < nlive; i += 2) {
        const int pa = slist[i], pb = (i + 1 < nlive) ? (int)slist[i + 1] : -1;
        PairParams P0, P1;
        load_pair(pa, P0);
        load_pair(pb < 0 ? pa : pb, P1);
        if (pb < 0) P1.c = dup(INFINITY);   // no second pair: q' = inf, e = 0
        uint32_t nz0 = 0u, nz1 = 0u;   // OR of the bits of e: nonzero iff some e is
#pragma unroll
        for (int p = 0; p < PT_P; ++p) {
            const float2 nq0 = neg_logit2(P0, X[p][0], X[p][1], X[p][2]);
            const float2 nq1 = neg_logit2(P1, X[p][0], X[p][1], X[p][2]);
            const float2 e0 = f2(ex2_approx(-nq0.x), ex2_approx(-nq0.y));
            const float2 e1 = f2(ex2_approx(-nq1.x), ex2_approx(-nq1.y));
            tot[p] = add2(tot[p], add2(e0, e1));
            if (STATS) {
                nz0 |= __float_as_uint(e0.x) | __float_as_uint(e0.y);
                nz1 |= __float_as_uint(e1.x) | __float_as_uint(e1.y);
            }
        }
        if (STATS) {
            const bool v0 = __ballot_sync(FULL, nz0 != 0u) != 0u, v1 = __ballot_sync(FULL, nz1 != 0u) != 0u;
            if (lane == 0) {
                if (v0) smask[pa >> 5] |= 1u << (pa & 31);
                if (v1) smask[pb >> 5] |= 1u << (pb & 31);   // v1 implies pb >= 0
            }
        }
    }
    __syncwarp();

    // ---- totals (the block's warps add their sums in the same order), log-likelihood,
    // rare points
#pragma unroll
    for (int p = 0; p < PT_P; ++p) s_tot[warp][p][lane] = tot[p];
    pt_block_sync(blk);
    float2 pr[PT_P];   // (shift, 1 / total) per point
    double ll = 0.0;
    bool rare_any = false;
#pragma unroll
    for (int p = 0; p < PT_P; ++p) {
        pr[p] = f2(0.f, 0.f);
        if (!valid[p]) continue;
        float t = 0.f;
#pragma unroll
        for (int h = 0; h < PT_H; ++h) {
            const float2 u = s_tot[blk * PT_H + h][p][lane];
            t += u.x + u.y;
        }
        float sh = 0.f;
        if (!(t >= 0x1p-100f)) {
            // every component is > 100 binades below cmax at this point: the exact maximum
            rare_any = true;
            float mx = -INFINITY;
            for (int pp = 0; pp < npairs; ++pp) {
                PairParams P;
                load_pair(pp, P);
                const float2 nq = neg_logit2(P, X[p][0], X[p][1], X[p][2]);
                mx = fmaxf(mx, fmaxf(-nq.x, -nq.y));
            }
            if (!(mx > -INFINITY)) {
                set_error(a.st, GIRA_ERR_NUMERIC);
                continue;
            }
            float sm = 0.f;
            for (int pp = 0; pp < npairs; ++pp) {
                PairParams P;
                load_pair(pp, P);
                const float2 nq = neg_logit2(P, X[p][0], X[p][1], X[p][2]);
                sm += ex2_approx(-nq.x - mx) + ex2_approx(-nq.y - mx);
            }
            t = sm;
            sh = -mx;
        }
        pr[p] = f2(sh, __frcp_rn(t));
        const float lse2 = lg2_approx(t) + ref0 - sh;   // log2 sum_b pi_b N(x|b)
        if (half == 0) {   // (every warp of the block has the same totals)
            ll += (double)lse2;
            if (!STATS && a.per_point) a.per_point[base + 32 * p] = lse2 * LN2F;
        }
    }

    if (STATS) {
        __syncwarp();
        if (__any_sync(FULL, rare_any) && lane < nwords) {   // every evaluated pair of this warp
            const int lo = lane * 32;
            const uint32_t mine = PT_H == 1 ? 0xffffffffu : (half ? 0xaaaaaaaau : 0x55555555u);
            smask[lane] = mine & ((lo + 32 <= npairs) ? 0xffffffffu : (lo < npairs) ? ((1u << (npairs - lo)) - 1u) : 0u);
        }
        pt_block_sync(blk);   // the block's masks are final
        const int64_t gw = (int64_t)cta * PT_B + blk;
        const int64_t rows = a.pt_rows;
        if (half == 0 && lane < nwords) {
            uint32_t m = 0u;
#pragma unroll
            for (int h = 0; h < PT_H; ++h) m |= smask_all[(blk * PT_H + h) * nwords + lane];
            if (GIRA_IN(gw < rows, a.st)) a.masks[lane * rows + gw] = m;
        }
        if (lane == 0) {
            unsigned live = 0;
            for (int wd = 0; wd < nwords; ++wd) live += __popc(smask[wd]);
            s_pairs[warp][0] = (unsigned)nlive;
            s_pairs[warp][1] = live;
        }
        // ---- phase 2: this warp's live pairs; partials [rows][pairs][2 NSTAT], masks [nwords][rows]
        for (int wd = 0; wd < nwords; ++wd) {
            uint32_t m = smask[wd];
            while (m) {
                const int pp = wd * 32 + __ffs(m) - 1;
                m &= m - 1u;
                PairParams P;
                load_pair(pp, P);
                float2 S[NSTAT];
#pragma unroll
                for (int s2 = 0; s2 < NSTAT; ++s2) S[s2] = f2(0.f, 0.f);
#pragma unroll
                for (int p = 0; p < PT_P; ++p) {
                    float2 y0, y1, y2;
                    const float2 nq = neg_logit2_y(P, X[p][0], X[p][1], X[p][2], y0, y1, y2);
                    const float2 e = f2(ex2_approx(pr[p].x - nq.x), ex2_approx(pr[p].x - nq.y));
                    const float2 g = mul2(e, dup(pr[p].y));   // pr = 0 for invalid points: g = 0
                    const float2 g0 = mul2(g, y0), g1 = mul2(g, y1), g2 = mul2(g, y2);
                    S[0] = add2(S[0], g);
                    S[1] = add2(S[1], g0);
                    S[2] = add2(S[2], g1);
                    S[3] = add2(S[3], g2);
                    S[4] = fma2(g0, y0, S[4]);
                    S[5] = fma2(g0, y1, S[5]);
                    S[6] = fma2(g0, y2, S[6]);
                    S[7] = fma2(g1, y1, S[7]);
                    S[8] = fma2(g1, y2, S[8]);
                    S[9] = fma2(g2, y2, S[9]);
                }
                int v;
                const float r = pt_warp_reduce20(S, lane, &v);
                const int b = 2 * pp + (v >= NSTAT ? 1 : 0);
                if ((lane & 7) < 5 && b < a.k && GIRA_IN(gw < rows, a.st))
                    a.partials[(size_t)gw * pt_row_floats(a.k) + (size_t)pp * 2 * NSTAT + v] = r;
            }
        }
    }
    // the CTA's log-likelihood: lanes, then warps in order
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) ll += __shfl_xor_sync(FULL, ll, o);
    if (lane == 0) s_ll[warp] = ll;
    __syncthreads();
    if (threadIdx.x == 0) {
        double v = s_ll[0];
        for (int w = 1; w < PT_W; ++w) v += s_ll[w];
        if (GIRA_IN(cta < (a_in.units ? a.pt_rows / PT_B : (int64_t)gridDim.x), a.st)) a.ll_partials[cta] = v * LN2;
        if (STATS) {
            unsigned long long near = 0, live = 0;
            for (int w = 0; w < PT_W; ++w) {
                near += s_pairs[w][0];
                live += s_pairs[w][1];
            }
            atomicAdd(&a.st->pairs_near, near);
            atomicAdd(&a.st->pairs_live, live);
            if (a_in.cta_key) {   // the CTA's slowest warp, in units of a point's pair evaluations
                unsigned wmax = 0;
                for (int w = 0; w < PT_W; ++w)
                    wmax = max(wmax, PT_COST_NEAR * s_pairs[w][0] + PT_COST_LIVE * s_pairs[w][1]);
                if (GIRA_IN(cta < (int)gridDim.x, a.st)) a_in.cta_key[cta] = work_key(wmax);
            }
        }
    }
}

}  // namespace

// Pairs the parameter buffer holds for k components (whole CTA tables of 32 pairs up to
// 64 components, 64 pairs beyond; the extra slots are padding components).
int params_pairs_padded(int k) { return k <= 64 ? 32 : (k + 127) / 128 * 64; }

namespace {
thread_local std::string t_estep_name;
thread_local const void* t_estep_fn = nullptr;
}  // namespace

// The launched function's name as the runtime reports it, demangled, without
// its namespaces and parameter list.
void note_estep_kernel(const void* fn) {
    if (fn == t_estep_fn) return;
    t_estep_fn = fn;
    const char* raw = nullptr;
    if (cudaFuncGetName(&raw, fn) != cudaSuccess || !raw) {
        cudaGetLastError();
        t_estep_name = "estep_kernel";
        return;
    }
    int ok = -1;
    char* dem = abi::__cxa_demangle(raw, nullptr, nullptr, &ok);
    std::string name = (ok == 0 && dem) ? dem : raw;
    std::free(dem);
    size_t at = name.find("estep_pt_kernel<");
    if (at == std::string::npos) at = name.find("estep_adjoint_kernel<");
    if (at == std::string::npos) at = name.find("estep_reach_kernel<");
    if (at == std::string::npos) at = name.find("estep4_dense_kernel<");
    if (at != std::string::npos) name = name.substr(at);
    const size_t par = name.rfind(">(");
    if (par != std::string::npos) name = name.substr(0, par + 1);
    t_estep_name = name;
}

const char* last_estep_kernel() { return t_estep_name.c_str(); }

int estep_pt_grid(int64_t n) { return (int)std::max<int64_t>(1, (n + PT_PTS - 1) / PT_PTS); }
int estep_pt_rows(int grid) { return grid * PT_B; }
int estep_pt_row_floats(int k) { return pt_row_floats(k); }
int estep_pt_mask_words(int k) { return pt_pairs(k) / 32; }

cudaError_t launch_estep_pt(const EStepLaunch& a, bool stats, int grid, cudaStream_t s, bool pdl) {
    void* args[] = {(void*)&a};
    const void* fn = stats ? (const void*)estep_pt_kernel<true> : (const void*)estep_pt_kernel<false>;
    note_estep_kernel(fn);
    const size_t smem = pt_smem_bytes(a.k);
    cudaError_t e = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    PdlConfig c(dim3(grid), dim3(32 * PT_W), smem, s, pdl);
    return cudaLaunchKernelExC(&c.cfg, fn, args);
}

cudaError_t launch_estep_pt_units(const EStepLaunch& a, bool stats, int nunits, int kmax, cudaStream_t s) {
    void* args[] = {(void*)&a};
    const void* fn = stats ? (const void*)estep_pt_kernel<true> : (const void*)estep_pt_kernel<false>;
    note_estep_kernel(fn);
    const size_t smem = pt_smem_bytes(kmax);
    cudaError_t e = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    return cudaLaunchKernel(fn, dim3(nunits), dim3(32 * PT_W), args, smem, s);
}

int estep_pt_points() { return PT_PTS; }
int estep_pt_blocks() { return PT_B; }

// ------------------------------------------------------------------ pack + padding
namespace {
// Point i, packed; returns whether it is finite.
__device__ __forceinline__ bool pack_point(const float* __restrict__ p3, int64_t i, float4* __restrict__ p4,
                                           float4* __restrict__ p8) {
    const float x = p3[3 * i], y = p3[3 * i + 1], z = p3[3 * i + 2];
    if (p4) p4[i] = make_float4(x, y, z, 0.f);
    if (p8) {
        p8[2 * i] = make_float4(x, x, y, y);
        p8[2 * i + 1] = make_float4(z, z, 0.f, 0.f);
    }
    return isfinite(x) && isfinite(y) && isfinite(z);
}

__global__ void pack_kernel(const float* __restrict__ p3, int64_t n, float4* __restrict__ p4,
                            float4* __restrict__ p8, DeviceState* st) {
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n && !pack_point(p3, i, p4, p8)) set_error(st, GIRA_ERR_NONFINITE_INPUT);
}

__device__ __forceinline__ void pad_slot(float* params, int b) {
    float* base = params + (size_t)(b >> 1) * PAIR_FLOATS + (b & 1);
    for (int s = 0; s < PAIR_FLOATS / 2; ++s) base[2 * s] = 0.f;
    base[2 * SLOT_C] = -INFINITY;
}

// One block per instance: the padding component slots k .. 2 * npairs - 1 of its block.
__global__ void fill_padding_batched_kernel(float* params, const BatchInst* __restrict__ insts,
                                            const int* __restrict__ npairs_of) {
    const BatchInst I = insts[blockIdx.x];
    const int slots = 2 * npairs_of[blockIdx.x];
    for (int b = I.k + threadIdx.x; b < slots; b += blockDim.x) pad_slot(params + I.par_off, b);
}

__global__ void fill_padding_kernel(float* params, int k, int npairs_pad) {
    int b = blockIdx.x * blockDim.x + threadIdx.x;   // component slot
    if (b >= 2 * npairs_pad || b < k) return;
    pad_slot(params, b);
}
}  // namespace

// Every point of a batch; the instance of point i (for the error flag) by binary
// search over the offsets (batch + 1 entries).
__global__ void pack_batched_kernel(const float* __restrict__ p3, int64_t n, const int64_t* __restrict__ offsets,
                                    int batch, float4* __restrict__ p4, float4* __restrict__ p8, DeviceState* states) {
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const float x = p3[3 * i], y = p3[3 * i + 1], z = p3[3 * i + 2];
    if (!(isfinite(x) && isfinite(y) && isfinite(z))) {
        int lo = 0, hi = batch;   // offsets[lo] <= i < offsets[hi]
        while (hi - lo > 1) {
            const int mid = (lo + hi) >> 1;
            if (offsets[mid] <= i) lo = mid; else hi = mid;
        }
        set_error(states + lo, GIRA_ERR_NONFINITE_INPUT);
    }
    if (p4) p4[i] = make_float4(x, y, z, 0.f);
    if (p8) {
        p8[2 * i] = make_float4(x, x, y, y);
        p8[2 * i + 1] = make_float4(z, z, 0.f, 0.f);
    }
}

cudaError_t launch_pack_batched(const float* pts3, int64_t n, const int64_t* offsets, int batch, float4* pts4,
                                float4* pts8, DeviceState* states, cudaStream_t s) {
    pack_batched_kernel<<<(unsigned)((n + 255) / 256), 256, 0, s>>>(pts3, n, offsets, batch, pts4, pts8, states);
    return cudaGetLastError();
}

cudaError_t launch_pack(const float* pts3, int64_t n, float4* pts4, float4* pts8, DeviceState* st, cudaStream_t s) {
    int64_t blocks = (n + 255) / 256;
    pack_kernel<<<(unsigned)blocks, 256, 0, s>>>(pts3, n, pts4, pts8, st);
    return cudaGetLastError();
}

cudaError_t launch_fill_padding(float* params, int k, int npairs_pad, cudaStream_t s) {
    int slots = 2 * npairs_pad;
    fill_padding_kernel<<<(slots + 127) / 128, 128, 0, s>>>(params, k, npairs_pad);
    return cudaGetLastError();
}

// ------------------------------------------------------------------ log-likelihood reduce
namespace {
// The sum of n partials by one block, in an order that depends on n alone (a fit and a batch
// give the same bits); valid in thread 0.  1,080 partials: 6.2 us by one warp, 4.5 us by eight.
constexpr int LLR_THREADS = 256;
__device__ double ll_block_sum(const double* __restrict__ llp, int n) {
    __shared__ double s_w[LLR_THREADS / 32];
    double v = 0.0;
    for (int c = threadIdx.x; c < n; c += LLR_THREADS) v += llp[c];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(FULL, v, o);
    if ((threadIdx.x & 31) == 0) s_w[threadIdx.x >> 5] = v;
    __syncthreads();
    v = s_w[0];
    if (threadIdx.x == 0)
        for (int w = 1; w < LLR_THREADS / 32; ++w) v += s_w[w];
    return v;
}

__global__ void __launch_bounds__(LLR_THREADS) ll_reduce_batched_kernel(const double* __restrict__ llp,
                                                                        const BatchInst* __restrict__ insts,
                                                                        DeviceState* states) {
    const BatchInst I = insts[blockIdx.x];
    const double v = ll_block_sum(llp + I.ll_off, I.ctas);
    if (threadIdx.x == 0) states[blockIdx.x].ll_sum = v;
}

__global__ void __launch_bounds__(LLR_THREADS) ll_reduce_kernel(const double* __restrict__ llp, int grid,
                                                                DeviceState* st) {
    if (st->error) return;   // uniform: nothing sets it now
    const double v = ll_block_sum(llp, grid);
    if (threadIdx.x == 0) st->ll_sum = v;
}
}  // namespace

cudaError_t launch_ll_reduce(const double* ll_partials, int grid, DeviceState* st, cudaStream_t s) {
    ll_reduce_kernel<<<1, LLR_THREADS, 0, s>>>(ll_partials, grid, st);
    return cudaGetLastError();
}

// ------------------------------------------------------------------ FP64 M-step
namespace {

constexpr int FIN_CPB = 2;          // components per block: spreads the binary64 work over SMs
constexpr int FIN_SPLIT_CTA = 16;   // per-CTA partials: one output summed in 16 fixed slices
constexpr int FIN_SPLIT = 64;       // per-warp rows: one float4 of outputs summed in 64 fixed slices
constexpr int FIN_THREADS = FIN_CPB * NSTAT * FIN_SPLIT_CTA;   // 320
constexpr int ORDER_THREADS = 1024;   // order_components_kernel: one block
constexpr int ORDER_MAX_K = 8192;     // keys in dynamic shared memory (64 KB)

// ---- the parameter build, shared by the scalar and the warp-parallel forms.
// Every helper fixes its binary64 operations (explicit rounding intrinsics, no
// contraction left to the compiler), so both forms give the same bits.

// Cholesky Sigma = L L^T of c = (00, 01, 02, 11, 12, 22) by Schur complements,
// in terms of the pivots' reciprocal square roots:
//   u = a00^-1/2, r0 = u^2, h0 = a01 r0,
//   s11 = a11 - h0 a01, s12 = a12 - h0 a02, s22 = a22 - (a02 r0) a02,
//   v = s11^-1/2, t = s12 v^2, a22' = s22 - t s12, z = a22'^-1/2, g = a02 - a01 t;
// then P = L^-1 has P00 = u, P11 = v, P22 = z, P10 = -h0 v, P21 = -t z,
// P20 = -(r0 g) z, and prod_j P_jj = u v z.  pd: every pivot positive.
struct CholInv {
    double u, v, z, r0, h0, t, g;
    bool pd;
};

__device__ __forceinline__ CholInv chol_inv(const double c[6]) {
    CholInv k;
    k.u = rsqrt(c[0]);
    k.r0 = __dmul_rn(k.u, k.u);
    k.h0 = __dmul_rn(c[1], k.r0);
    const double h1 = __dmul_rn(c[2], k.r0);
    const double s11 = __fma_rn(-k.h0, c[1], c[3]);
    const double s12 = __fma_rn(-k.h0, c[2], c[4]);
    const double s22 = __fma_rn(-h1, c[2], c[5]);
    k.v = rsqrt(s11);
    k.t = __dmul_rn(s12, __dmul_rn(k.v, k.v));
    const double a22 = __fma_rn(-k.t, s12, s22);
    k.z = rsqrt(a22);
    k.g = __fma_rn(-c[1], k.t, c[2]);
    k.pd = c[0] > 0.0 && s11 > 0.0 && a22 > 0.0;
    return k;
}

constexpr double ALPHA = 0.84932180028801904272;   // sqrt(log2(e) / 2)

// Entry e of P' = alpha L^-1 in the order (00, 10, 11, 20, 21, 22), as
// alpha ((A B) C) with (A, B, C) = (u, 1, 1), (h0, v, -1), (v, 1, 1), (r0, g, -z),
// (t, z, -1), (z, 1, 1): the same three products for every entry.
__device__ __forceinline__ double chol_q(const CholInv& k, int e) {
    const double A = e == 0 ? k.u : e == 1 ? k.h0 : e == 2 ? k.v : e == 3 ? k.r0 : e == 4 ? k.t : k.z;
    const double B = e == 1 ? k.v : e == 3 ? k.g : e == 4 ? k.z : 1.0;
    const double C = e == 1 || e == 4 ? -1.0 : e == 3 ? -k.z : 1.0;
    return __dmul_rn(ALPHA, __dmul_rn(__dmul_rn(A, B), C));
}

// b_i = -(P' mu)_i from the row (a0, a1, a2) of P' (zeros above the diagonal).
__device__ __forceinline__ double bias_row(double a0, double a1, double a2, const double mu[3]) {
    return -__fma_rn(a2, mu[2], __fma_rn(a1, mu[1], __dmul_rn(a0, mu[0])));
}

// c = log2(w prod_j P_jj) - (3/2) log2(2 pi) in binary32: the exponent of
// x = w u v z exactly, log2f of its significand rounded to 24 bits (error a
// few 1e-8), the constant 4 - (3/2) log2(2 pi) = 0.0227558057915218 folded in.
__device__ __forceinline__ float log2_norm(double w, const CholInv& k) {
    const double x = __dmul_rn(w, __dmul_rn(__dmul_rn(k.u, k.v), k.z));
    if (!(x >= DBL_MIN && x <= DBL_MAX)) return (float)(log2(x) - 3.9772441942084782);
    const unsigned long long bits = (unsigned long long)__double_as_longlong(x);
    const int e = (int)((bits >> 52) & 0x7ffu) - 1023;
    const unsigned int m24 = (unsigned int)(((bits & 0xfffffffffffffull) + (1ull << 28)) >> 29);   // 0 .. 2^23
    const float m = __int_as_float((127 << 23) + (int)m24);   // the significand in [1, 2]
    return __fadd_rn((float)(e - 4), __fadd_rn(log2f(m), 0.0227558057915218f));
}

// alpha^2 / lambda_max(Sigma), lowered by 1e-4 relative: a lower bound of
// sigma_min(P')^2 for the E-step's reach test.  lambda_max by the trigonometric
// solution of the characteristic cubic of a symmetric 3x3 matrix in binary32
// (error a few ulps), raised by 1e-4 relative; trace(Sigma) where the cubic is
// degenerate; never below the largest diagonal entry.
__device__ __forceinline__ float sigma_min_sq_bound(const float a[6]) {
    const float a00 = a[0], a01 = a[1], a02 = a[2], a11 = a[3], a12 = a[4], a22 = a[5];
    const float tr3 = (a00 + a11 + a22) * (1.f / 3.f);
    const float e0 = a00 - tr3, e1 = a11 - tr3, e2 = a22 - tr3;
    const float p2 = e0 * e0 + e1 * e1 + e2 * e2 + 2.f * (a01 * a01 + a02 * a02 + a12 * a12);
    float lmax = 3.f * tr3;
    if (p2 > 1e-30f) {
        const float pp = sqrtf(p2 * (1.f / 6.f)), ip = 1.f / pp;
        const float b00 = e0 * ip, b11 = e1 * ip, b22 = e2 * ip, b01 = a01 * ip, b02 = a02 * ip, b12 = a12 * ip;
        const float det = b00 * (b11 * b22 - b12 * b12) - b01 * (b01 * b22 - b12 * b02) + b02 * (b01 * b12 - b11 * b02);
        const float r = fminf(1.f, fmaxf(-1.f, 0.5f * det));
        const float trig = tr3 + 2.f * pp * cosf(acosf(r) * (1.f / 3.f));
        if (trig == trig) lmax = fminf(lmax, trig * (1.f + 1e-4f));
    }
    lmax = fmaxf(lmax, fmaxf(a00, fmaxf(a11, a22)) * (1.f + 1e-4f));
    return (float)(ALPHA * ALPHA) / lmax * (1.f - 1e-4f);
}

// From (w, mu, Sigma) in binary64 to the E-step parameters of component b
// (scalar form; the EM finalize runs the same helpers lane-parallel).
// Returns false (and flags GIRA_ERR_NOT_PD) if a pivot is not positive.
// report: the caller's index of the component (differs from b when the fit
// holds its components in another order).
__device__ bool build_component(int b, double w, const double mu[3], const double c[6], float* params,
                                float4* shift4, double* model64, DeviceState* st, int report) {
    const CholInv k = chol_inv(c);
    if (!k.pd) {
        atomicMin(&st->bad_component, report);
        set_error(st, GIRA_ERR_NOT_PD);
        return false;
    }
    double q[6];
    for (int e = 0; e < 6; ++e) q[e] = chol_q(k, e);
    float* base = params + (size_t)(b >> 1) * PAIR_FLOATS + (b & 1);
    for (int i = 0; i < 6; ++i) base[2 * (SLOT_P + i)] = (float)q[i];
    base[2 * (SLOT_B + 0)] = (float)bias_row(q[0], 0.0, 0.0, mu);
    base[2 * (SLOT_B + 1)] = (float)bias_row(q[1], q[2], 0.0, mu);
    base[2 * (SLOT_B + 2)] = (float)bias_row(q[3], q[4], q[5], mu);
    base[2 * SLOT_C] = log2_norm(w, k);
    const float m32[3] = {(float)mu[0], (float)mu[1], (float)mu[2]};
    for (int i = 0; i < 3; ++i) base[2 * (SLOT_NMU + i)] = -m32[i];
    base[2 * SLOT_W] = (float)w;
    const float c32[6] = {(float)c[0], (float)c[1], (float)c[2], (float)c[3], (float)c[4], (float)c[5]};
    base[2 * SLOT_S] = sigma_min_sq_bound(c32);
    shift4[b] = make_float4(m32[0], m32[1], m32[2], 0.f);
    double* m = model64 + (size_t)b * MODEL;
    m[0] = w;
    m[1] = mu[0]; m[2] = mu[1]; m[3] = mu[2];
    for (int i = 0; i < 6; ++i) m[4 + i] = c[i];
    return true;
}

// Compensated binary32 accumulation (Knuth's TwoSum: the rounding error of each
// addition, exact under round-to-nearest, is carried in e).
__device__ __forceinline__ void two_sum_acc(float& s, float& e, float x) {
    const float t = __fadd_rn(s, x);
    const float bp = __fsub_rn(t, s);
    const float err = __fadd_rn(__fsub_rn(s, __fsub_rn(t, bp)), __fsub_rn(x, bp));
    s = t;
    e = __fadd_rn(e, err);
}

// Per-component binary64 work area of the finalize (shared memory), in doubles.
constexpr int FW = 64;
constexpr int W_S = 0;      // S0, S1[3], S2[6]
constexpr int W_QS = 10;    // P' (00,10,11,20,21,22) and the shift s[3]; later the new P' and b
constexpr int W_R = 19;     // 1/q00, 1/q11, 1/q22, 1/N_b
constexpr int W_T = 23;     // ybar[3], m10, m21
constexpr int W_M = 28;     // M = P'^-1 (3x3 row-major; the identity for one-hot statistics)
constexpr int W_CY = 37;    // C (3x3, both halves)
constexpr int W_MU = 46;    // the new mean
constexpr int W_MC = 49;    // M C (3x3)
constexpr int W_C = 58;     // the new Sigma (00,01,02,11,12,22)
constexpr int FF = 20;      // binary32 copies per component: P'[6], b[3], mu[3], w, Sigma[6]

// The statistics of the pair of components b0, b0 + 1 (b0 even) from the per-warp
// partial rows of the point-stationary E-step ([rows][pairs][2 NSTAT] binary32, a
// pair's 20 values 80 contiguous bytes): the rows whose live mask has the pair's bit
// are listed in row order (one block scan per segment of FIN_SEG rows, each thread
// ranking a contiguous run of rows).  Thread (c, q) = (t / 64, t % 64) sums float4 c
// of the pair's values (outputs 4c .. 4c + 3; output o is component o / NSTAT,
// statistic o % NSTAT) over the q-th of FIN_SPLIT fixed contiguous slices of the list
// in compensated binary32; a fixed butterfly of compensated additions joins the 32
// slices of a warp, then the two warps of c in order, and each (sum, error) becomes
// one binary64 value in W.  The list depends only on the masks, so the order of every
// addition is fixed.  Call with every thread of the block; s_skip (set by thread 0
// before the call) is read after the first barrier, and a skipped block returns false
// before touching W.
constexpr int FIN_SEG = 4096;
static_assert(FIN_THREADS == 5 * 64 && FIN_SPLIT == 64 && 2 * NSTAT == 20, "five float4 of a pair, 64 slices each");
__device__ bool reduce_partials_masked(const float* __restrict__ partials, int rows, int row_floats,
                                       const uint32_t* __restrict__ masks, int b0, int nout, double (*W)[FW],
                                       const int* s_skip, DeviceState* st) {
    __shared__ uint16_t s_list[FIN_SEG];
    __shared__ int s_wsum[FIN_THREADS / 32];
    __shared__ float s_hi[FIN_THREADS / 64][8];
    const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
    const int c = t >> 6, q = t & 63;
    const uint32_t* mrow = masks + (size_t)((b0 >> 1) >> 5) * rows;
    const uint32_t bit = 1u << ((b0 >> 1) & 31);
    const float4* src = reinterpret_cast<const float4*>(partials + (size_t)(b0 >> 1) * 2 * NSTAT) + c;
    const size_t stride4 = (size_t)row_floats / 4;
    float sum[4] = {0.f, 0.f, 0.f, 0.f}, err[4] = {0.f, 0.f, 0.f, 0.f};
    for (int seg0 = 0; seg0 < rows; seg0 += FIN_SEG) {
        const int seg1 = min(rows, seg0 + FIN_SEG);
        constexpr int RND = (FIN_SEG + FIN_THREADS - 1) / FIN_THREADS;
        const int per = (seg1 - seg0 + FIN_THREADS - 1) / FIN_THREADS;   // rows ranked by one thread
        const int r0 = seg0 + t * per;
        uint32_t live = 0u;   // bit u: row r0 + u is live
#pragma unroll
        for (int u = 0; u < RND; ++u) {
            const uint32_t mw = (u < per && r0 + u < seg1) ? __ldg(mrow + r0 + u) : 0u;
            if (mw & bit) live |= 1u << u;
        }
        const int cnt = __popc(live);
        int incl = cnt;   // inclusive scan of the counts over the warp
#pragma unroll
        for (int d = 1; d < 32; d <<= 1) {
            const int v = __shfl_up_sync(FULL, incl, d);
            if (lane >= d) incl += v;
        }
        if (lane == 31) s_wsum[warp] = incl;
        __syncthreads();
        if (*s_skip) return false;
        int off = incl - cnt, nl = 0;
#pragma unroll
        for (int w = 0; w < FIN_THREADS / 32; ++w) {
            const int cw = s_wsum[w];
            off += (w < warp) ? cw : 0;
            nl += cw;
        }
        for (uint32_t m = live; m; m &= m - 1u) {
            const int r = r0 + __ffs(m) - 1;
            if (GIRA_IN(off < FIN_SEG, st)) s_list[off] = (uint16_t)(r - seg0);
            ++off;
        }
        __syncthreads();
        const int c0 = q * nl / FIN_SPLIT, c1 = (q + 1) * nl / FIN_SPLIT;
        const float4* sseg = src + (size_t)seg0 * stride4;
        for (int i = c0; i < c1; i += 8) {   // eight float4 loads in flight
            float4 v[8];
#pragma unroll
            for (int u = 0; u < 8; ++u)
                v[u] = (i + u < c1 && GIRA_IN(s_list[i + u] < seg1 - seg0, st))
                           ? __ldcg(sseg + (size_t)s_list[i + u] * stride4) : make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
            for (int u = 0; u < 8; ++u) {
                if (i + u < c1) {
                    two_sum_acc(sum[0], err[0], v[u].x);
                    two_sum_acc(sum[1], err[1], v[u].y);
                    two_sum_acc(sum[2], err[2], v[u].z);
                    two_sum_acc(sum[3], err[3], v[u].w);
                }
            }
        }
        __syncthreads();   // the list is rebuilt for the next segment
    }
#pragma unroll
    for (int d = 16; d > 0; d >>= 1) {   // butterfly over the warp: the same totals in every lane
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            const float s2 = __shfl_xor_sync(FULL, sum[j], d), e2 = __shfl_xor_sync(FULL, err[j], d);
            float e = __fadd_rn(err[j], e2);
            two_sum_acc(sum[j], e, s2);
            err[j] = e;
        }
    }
    if ((warp & 1) && lane == 0) {   // the second warp of c: slices 32 .. 63
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            s_hi[c][j] = sum[j];
            s_hi[c][4 + j] = err[j];
        }
    }
    __syncthreads();
    if (!(warp & 1) && lane < 4) {
        const int j = lane;
        float sj = j == 0 ? sum[0] : j == 1 ? sum[1] : j == 2 ? sum[2] : sum[3];
        float ej = j == 0 ? err[0] : j == 1 ? err[1] : j == 2 ? err[2] : err[3];
        ej = __fadd_rn(ej, s_hi[c][4 + j]);
        two_sum_acc(sj, ej, s_hi[c][j]);
        const int o = 4 * c + j;
        if (o < nout) W[o / NSTAT][W_S + o % NSTAT] = __dadd_rn((double)sj, (double)ej);
    }
    return true;
}

// M-step (the standard full-covariance update) from shifted statistics:
//   N_b = S0 + 10 eps; with v = y = P'(x - s_b) (E-step partials, whitened) or
//   v = d = x - s_b (one-hot KInit statistics): vbar = S1 / N_b and the centred
//   second moment C = S2 / N_b - vbar vbar^T (S1 = N_b vbar); mu = s + M vbar and
//   Sigma = M C M^T + reg I with M = P'^-1 (whitened) or M = I (one-hot).  The
//   weight N_b is normalised by sum_a N_a where it is used (E-step reference,
//   model output).
struct FinArgs {
    const float* partials;     // [grid][k][NSTAT], or nullptr (then stats64)
    int grid;
    const double* llp;
    const double* stats64;
    float4* shift4;
    int k;
    int64_t n;
    double reg, tol;
    double* model64;
    float* params;
    double* trace;
    DeviceState* st;
    int iter, em;
    int ll_count;   // log-likelihood partials to sum (grid when 0)
    int do_ll;      // this launch's block 0 does the log-likelihood / convergence step
    const int* perm;   // slot b holds the caller's component perm[b] (nullptr: b)
    // point-stationary E-step: partial rows per block of points ([grid rows][pairs]
    // [2 NSTAT]), a pair's values valid only where the row's live mask ([nwords]
    // [grid rows]) has the pair's bit
    const uint32_t* masks;
    int nwords;
    // a single fit's CTA order: the launch's last block ranks the E-step's cta_grid
    // CTAs by cta_key into cta_perm[(iter & 1) * cta_grid ..] for iteration iter + 2
    const uint8_t* cta_key = nullptr;
    int* cta_perm = nullptr;
    int cta_grid = 0;
};

__device__ __forceinline__ int sym_i(int u) { return u < 3 ? 0 : (u < 5 ? 1 : 2); }   // (00,01,02,11,12,22)
__device__ __forceinline__ int sym_j(int u) { return u < 3 ? u : (u < 5 ? u - 2 : 2); }
__device__ __forceinline__ double dneg(double x) {   // sign flip on the integer pipe
    return __longlong_as_double(__double_as_longlong(x) ^ (long long)0x8000000000000000ull);
}

// The M-step and the parameter build of components b0 + h (h = 0, 1) by one
// warp: lanes 16 h .. 16 h + 15 take component b0 + h, and each stage computes
// its entries in parallel lanes, every entry by a fixed sequence of binary64
// operations (GB300 issues one binary64 warp instruction every 64 cycles per
// warp, whatever the number of active lanes, so a stage costs what one entry
// costs).  W[h][W_S ..] holds the statistics; pre is this lane's binary32 P'
// entry (l < 6) or shift coordinate (6 <= l < 9), loaded at the kernel's start.
__device__ void finalize_update_warp(const FinArgs& f, int b0, int nb, float pre, double (*W)[FW], float (*F)[FF]) {
    const int lane = threadIdx.x & 31, h = lane >> 4, l = lane & 15;
    const int b = b0 + h;
    const bool on = h < nb;
    double* w = W[h];
    const bool white = f.partials != nullptr;
    if (on && l < 9) w[W_QS + l] = (double)pre;
    __syncwarp();
    const double nbw = __dadd_rn(w[W_S], 10.0 * DBL_EPSILON);
    // the reciprocals of q00, q11, q22 (the diagonal of M) and of N_b
    if (on && l < 4) {
        const double x = l == 3 ? nbw : (white ? w[W_QS + (l == 0 ? 0 : (l == 1 ? 2 : 5))] : 1.0);
        w[W_R + l] = __drcp_rn(x);
    }
    __syncwarp();
    const double inv = w[W_R + 3];
    // vbar = S1 / N_b (l < 3); m10 = -q10 m00 m11 (l == 3), m21 = -q21 m11 m22 (l == 4)
    if (on && l < 5) {
        double A, B, C;
        if (l < 3) {
            A = w[W_S + 1 + l]; B = inv; C = 1.0;
        } else {
            const int j = l - 3;
            A = dneg(w[W_QS + (j == 0 ? 1 : 4)]); B = w[W_R + j]; C = w[W_R + j + 1];
        }
        w[W_T + l] = __dmul_rn(__dmul_rn(A, B), C);
    }
    __syncwarp();
    // C = S2 / N_b - vbar vbar^T (l < 6), m20 = -(q20 m00 + q21 m10) m22 (l == 6);
    // lanes 7 .. 14 place the other entries of M
    if (on && l < 7) {
        const int i = sym_i(l < 6 ? l : 0), j = sym_j(l < 6 ? l : 0);
        double A0, B0, A1, B1, C;
        if (l < 6) {
            A0 = w[W_S + 4 + l]; B0 = inv; A1 = dneg(w[W_T + i]); B1 = w[W_T + j]; C = 1.0;
        } else {
            A0 = w[W_QS + 3]; B0 = w[W_R + 0]; A1 = w[W_QS + 4]; B1 = w[W_T + 3]; C = dneg(w[W_R + 2]);
        }
        const double v = __dmul_rn(__fma_rn(A1, B1, __dmul_rn(A0, B0)), C);
        if (l < 6) {
            w[W_CY + 3 * i + j] = v;
            w[W_CY + 3 * j + i] = v;
        } else {
            w[W_M + 6] = white ? v : 0.0;
        }
    } else if (on && l < 15) {
        const int e = l - 7 + (l >= 13 ? 1 : 0);   // 0 .. 5, 7, 8
        double v;
        if (!white) v = (e == 0 || e == 4 || e == 8) ? 1.0 : 0.0;
        else v = e == 0 ? w[W_R + 0] : e == 3 ? w[W_T + 3] : e == 4 ? w[W_R + 1] : e == 7 ? w[W_T + 4]
                                     : e == 8 ? w[W_R + 2] : 0.0;
        w[W_M + e] = v;
    }
    __syncwarp();
    // mu = s + M vbar (l < 3); M C (3 <= l < 12)
    if (on && l < 12) {
        const int i = l < 3 ? l : (l - 3) / 3, j = l < 3 ? 0 : (l - 3) % 3;
        const int bs = l < 3 ? 1 : 3;
        const double* Bv = l < 3 ? w + W_T : w + W_CY + j;
        const double* Mi = w + W_M + 3 * i;
        const double c0 = l < 3 ? w[W_QS + 6 + l] : 0.0;
        const double v = __fma_rn(Mi[2], Bv[2 * bs], __fma_rn(Mi[1], Bv[bs], __fma_rn(Mi[0], Bv[0], c0)));
        if (l < 3) w[W_MU + l] = v;
        else w[W_MC + l - 3] = v;
    }
    __syncwarp();
    // Sigma = M C M^T + reg I (l < 6)
    if (on && l < 6) {
        const int i = sym_i(l), j = sym_j(l);
        const double* a = w + W_MC + 3 * i;
        const double* m = w + W_M + 3 * j;
        w[W_C + l] = __fma_rn(a[2], m[2], __fma_rn(a[1], m[1], __fma_rn(a[0], m[0], i == j ? f.reg : 0.0)));
    }
    __syncwarp();
    // the parameters (the scalar build_component's helpers, entries in parallel lanes)
    double c[6], mu[3];
    for (int e = 0; e < 6; ++e) c[e] = w[W_C + e];
    for (int i = 0; i < 3; ++i) mu[i] = w[W_MU + i];
    const CholInv k = chol_inv(c);
    const bool ok = on && k.pd;
    if (on && !k.pd && l == 0) {
        atomicMin(&f.st->bad_component, f.perm ? f.perm[b] : b);
        set_error(f.st, GIRA_ERR_NOT_PD);
    }
    if (ok && l < MODEL) {
        double* m = f.model64 + (size_t)b * MODEL;
        m[l] = l == 0 ? nbw : (l < 4 ? w[W_MU + l - 1] : w[W_C + l - 4]);
    }
    if (ok && l < 6) w[W_QS + l] = chol_q(k, l);
    __syncwarp();
    if (ok && l < 3) {
        const double* qq = w + W_QS;
        const double a0 = l == 0 ? qq[0] : (l == 1 ? qq[1] : qq[3]);
        const double a1 = l == 0 ? 0.0 : (l == 1 ? qq[2] : qq[4]);
        const double a2 = l == 2 ? qq[5] : 0.0;
        w[W_QS + 6 + l] = bias_row(a0, a1, a2, mu);
    }
    const float cc = log2_norm(nbw, k);
    __syncwarp();
    // binary32 copies: P'[6] and b[3] (W_QS ..), mu[3], w, Sigma[6]
    float* fc = F[h];
    if (ok) {
        for (int e = l; e < FF - 1; e += 16)
            fc[e] = (float)(e < 9 ? w[W_QS + e] : (e < 12 ? w[W_MU + e - 9] : (e == 12 ? nbw : w[W_C + e - 13])));
    }
    __syncwarp();
    if (ok) {
        float* base = f.params + (size_t)(b >> 1) * PAIR_FLOATS + (b & 1);
        static_assert(SLOT_B == SLOT_P + 6, "P' and b are consecutive slots");
        if (l < 9) base[2 * (SLOT_P + l)] = fc[l];
        else if (l == 9) base[2 * SLOT_C] = cc;
        else if (l < 13) base[2 * (SLOT_NMU + l - 10)] = -fc[l - 1];
        else if (l == 13) base[2 * SLOT_W] = fc[12];
        else if (l == 14) base[2 * SLOT_S] = sigma_min_sq_bound(fc + 13);
        else f.shift4[b] = make_float4(fc[9], fc[10], fc[11], 0.f);
    }
}

// The same for one component by one lane: every entry by the same sequence of operations, so
// the same bits.  A lane's chain is longer (8 us), but a binary64 instruction serves 32
// components where the half-warps above serve two.
__device__ void finalize_update_lane(const FinArgs& f, int b, bool white, const double* __restrict__ stats) {
    double S[NSTAT];
#pragma unroll
    for (int i = 0; i < NSTAT; ++i) S[i] = stats[i];
    float* base = f.params + (size_t)(b >> 1) * PAIR_FLOATS + (b & 1);
    const float4 sh = f.shift4[b];
    const double s0[3] = {(double)sh.x, (double)sh.y, (double)sh.z};
    const double nbw = __dadd_rn(S[0], 10.0 * DBL_EPSILON);
    const double inv = __drcp_rn(nbw);
    double M[3][3] = {{1.0, 0.0, 0.0}, {0.0, 1.0, 0.0}, {0.0, 0.0, 1.0}};
    if (white) {
        double q[6];
#pragma unroll
        for (int l = 0; l < 6; ++l) q[l] = (double)base[2 * (SLOT_P + l)];
        const double r0 = __drcp_rn(q[0]), r1 = __drcp_rn(q[2]), r2 = __drcp_rn(q[5]);
        M[0][0] = r0;
        M[1][1] = r1;
        M[2][2] = r2;
        M[1][0] = __dmul_rn(__dmul_rn(dneg(q[1]), r0), r1);
        M[2][1] = __dmul_rn(__dmul_rn(dneg(q[4]), r1), r2);
        M[2][0] = __dmul_rn(__fma_rn(q[4], M[1][0], __dmul_rn(q[3], r0)), dneg(r2));
    }
    double vb[3], C[3][3], mu[3], MC[3][3], c[6];
#pragma unroll
    for (int i = 0; i < 3; ++i) vb[i] = __dmul_rn(S[1 + i], inv);
#pragma unroll
    for (int l = 0; l < 6; ++l) {
        const int i = l < 3 ? 0 : (l < 5 ? 1 : 2), j = l < 3 ? l : (l < 5 ? l - 2 : 2);
        C[i][j] = C[j][i] = __fma_rn(dneg(vb[i]), vb[j], __dmul_rn(S[4 + l], inv));
    }
#pragma unroll
    for (int i = 0; i < 3; ++i) {
        mu[i] = __fma_rn(M[i][2], vb[2], __fma_rn(M[i][1], vb[1], __fma_rn(M[i][0], vb[0], s0[i])));
#pragma unroll
        for (int j = 0; j < 3; ++j)
            MC[i][j] = __fma_rn(M[i][2], C[2][j], __fma_rn(M[i][1], C[1][j], __fma_rn(M[i][0], C[0][j], 0.0)));
    }
#pragma unroll
    for (int l = 0; l < 6; ++l) {
        const int i = l < 3 ? 0 : (l < 5 ? 1 : 2), j = l < 3 ? l : (l < 5 ? l - 2 : 2);
        c[l] = __fma_rn(MC[i][2], M[j][2], __fma_rn(MC[i][1], M[j][1],
                                                    __fma_rn(MC[i][0], M[j][0], i == j ? f.reg : 0.0)));
    }
    const CholInv k = chol_inv(c);
    if (!k.pd) {
        atomicMin(&f.st->bad_component, f.perm ? f.perm[b] : b);
        set_error(f.st, GIRA_ERR_NOT_PD);
        return;
    }
    double* m = f.model64 + (size_t)b * MODEL;
    m[0] = nbw;
#pragma unroll
    for (int i = 0; i < 3; ++i) m[1 + i] = mu[i];
#pragma unroll
    for (int l = 0; l < 6; ++l) m[4 + l] = c[l];
    double q[6];
#pragma unroll
    for (int l = 0; l < 6; ++l) {
        q[l] = chol_q(k, l);
        base[2 * (SLOT_P + l)] = (float)q[l];
    }
    base[2 * SLOT_B] = (float)bias_row(q[0], 0.0, 0.0, mu);
    base[2 * (SLOT_B + 1)] = (float)bias_row(q[1], q[2], 0.0, mu);
    base[2 * (SLOT_B + 2)] = (float)bias_row(q[3], q[4], q[5], mu);
    base[2 * SLOT_C] = log2_norm(nbw, k);
    const float m32[3] = {(float)mu[0], (float)mu[1], (float)mu[2]};
#pragma unroll
    for (int i = 0; i < 3; ++i) base[2 * (SLOT_NMU + i)] = -m32[i];
    base[2 * SLOT_W] = (float)nbw;
    const float c32[6] = {(float)c[0], (float)c[1], (float)c[2], (float)c[3], (float)c[4], (float)c[5]};
    base[2 * SLOT_S] = sigma_min_sq_bound(c32);
    f.shift4[b] = make_float4(m32[0], m32[1], m32[2], 0.f);
}

// Components blk * FIN_CPB .. of one fit; block index blk == 0 also does the
// log-likelihood, trace and convergence of an EM iteration.
// sums != nullptr: only the statistics' sums, to sums[component][NSTAT].
__device__ void reduce_finalize_body(const FinArgs& f, int blk, double* sums = nullptr) {
    __shared__ double W[FIN_CPB][FW];
    __shared__ float F[FIN_CPB][FF];
    __shared__ int s_skip;
    static_assert(FIN_CPB == 2, "one half-warp per component in the update");
    const int t = threadIdx.x;
    const int b0 = blk * FIN_CPB;
    const int nb = min(FIN_CPB, f.k - b0);
    const int nout = nb * NSTAT;
    float pre = 0.f;   // warp 0: this lane's binary32 P' entry or shift coordinate, loaded early
    if (t < 32) {
        const int h = t >> 4, l = t & 15, b = b0 + h;
        if (h < nb && l < 9) {
            if (l < 6) {
                pre = f.partials ? f.params[(size_t)(b >> 1) * PAIR_FLOATS + (b & 1) + 2 * (SLOT_P + l)] : 0.f;
            } else {
                const float4 sh = f.shift4[b];
                pre = l == 6 ? sh.x : (l == 7 ? sh.y : sh.z);
            }
        }
    }
    if (t == 0) s_skip = (f.em && f.iter > f.st->stop_after) || f.st->error != 0;
    if (f.partials) {
        if (!reduce_partials_masked(f.partials, f.grid, pt_row_floats(f.k), f.masks, b0, nout, W, &s_skip, f.st))
            return;
    } else {
        __syncthreads();
        if (s_skip) return;
        if (t < nout) W[t / NSTAT][W_S + t % NSTAT] = f.stats64[(size_t)b0 * NSTAT + t];
    }
    __syncthreads();
    if (sums) {
        if (t < nout) sums[(size_t)b0 * NSTAT + t] = W[t / NSTAT][W_S + t % NSTAT];
    } else if (t < 32) {
        finalize_update_warp(f, b0, nb, pre, W, F);
        if (t == 0 && b0 == 0) f.st->w_raw = 1;
    }
    if (f.em && f.do_ll && blk == 0 && t >= 32) {   // warps 1 ..: log-likelihood, trace, convergence
        __shared__ double s_llw[FIN_THREADS / 32];
        const int lane = t & 31, w = t >> 5;
        double v = 0.0;
        const int nll = f.ll_count ? f.ll_count : f.grid;
        for (int c = t - 32; c < nll; c += FIN_THREADS - 32) v += f.llp[c];
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(FULL, v, o);
        if (lane == 0) s_llw[w] = v;
        asm volatile("bar.sync 1, %0;" ::"n"(FIN_THREADS - 32) : "memory");   // warps 1 .. only
        if (t == 32) {
            v = 0.0;
            for (int u = 1; u < FIN_THREADS / 32; ++u) v += s_llw[u];
            DeviceState* st = f.st;
            st->ll_sum = v;
            const double ll = v / (double)f.n;
            f.trace[f.iter - 1] = ll;
            if (f.iter > 1 && fabs(ll - st->prev_ll) < f.tol) st->stop_after = f.iter;
            st->prev_ll = ll;
            st->iters_done = f.iter;
        }
    }
}

// The E-step's CTA order for iteration f.iter + 2: descending work key, ties in
// index order (a counting sort: position = keys above + equal keys before).  The
// order changes only which SM runs which point blocks when, never a result.
__device__ void order_ctas(const FinArgs& f) {
    __shared__ int s_above[256], s_run[256];
    __shared__ uint16_t s_wc[FIN_THREADS / 32][256];
    const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
    const int grid = f.cta_grid;
    int* out = f.cta_perm + (size_t)(f.iter & 1) * grid;
    for (int b = t; b < 256; b += FIN_THREADS) s_above[b] = s_run[b] = 0;
    __syncthreads();
    for (int i = t; i < grid; i += FIN_THREADS) atomicAdd(&s_above[f.cta_key[i]], 1);
    __syncthreads();
    if (warp == 0) {   // s_above[b] = number of keys above b (8 buckets per lane, from the top)
        int v[8], tot = 0;
#pragma unroll
        for (int u = 0; u < 8; ++u) {
            v[u] = s_above[255 - (lane * 8 + u)];
            tot += v[u];
        }
        int incl = tot;
#pragma unroll
        for (int d = 1; d < 32; d <<= 1) {
            const int x = __shfl_up_sync(FULL, incl, d);
            if (lane >= d) incl += x;
        }
        __syncwarp();
        int run = incl - tot;
#pragma unroll
        for (int u = 0; u < 8; ++u) {
            s_above[255 - (lane * 8 + u)] = run;
            run += v[u];
        }
    }
    __syncthreads();
    for (int c0 = 0; c0 < grid; c0 += FIN_THREADS) {
        const int i = c0 + t;
        const int key = i < grid ? (int)f.cta_key[i] : -1;
        const unsigned peers = __match_any_sync(FULL, key);
        const int rank = __popc(peers & ((1u << lane) - 1u));
        for (int b = lane; b < 256; b += 32) s_wc[warp][b] = 0;
        __syncwarp();
        if (key >= 0 && rank == 0) s_wc[warp][key] = (uint16_t)__popc(peers);
        __syncthreads();
        if (key >= 0) {
            int pos = s_above[key] + s_run[key] + rank;
            for (int w = 0; w < warp; ++w) pos += s_wc[w][key];
            if (GIRA_IN(pos < grid, f.st)) out[pos] = i;
        }
        __syncthreads();
        for (int b = t; b < 256; b += FIN_THREADS) {
            int add = 0;
            for (int w = 0; w < FIN_THREADS / 32; ++w) add += s_wc[w][b];
            s_run[b] += add;
        }
        __syncthreads();
    }
}

__global__ void __launch_bounds__(FIN_THREADS) reduce_finalize_kernel(const FinArgs f) {
    pdl_wait();         // the E-step's partials (dependent launch)
    pdl_allow_next();   // the next E-step may stage its points meanwhile
    if (f.cta_key && blockIdx.x == gridDim.x - 1) {
        order_ctas(f);
        return;
    }
    reduce_finalize_body(f, blockIdx.x);
}

// Every instance of a batch: block (instance i, index j) finalizes components
// j * FIN_CPB .. of instance i from its own partials, into its own state.
__global__ void __launch_bounds__(FIN_THREADS) reduce_finalize_batched_kernel(const FinArgs base,
                                                                              const BatchInst* __restrict__ insts,
                                                                              const int2* __restrict__ blocks,
                                                                              DeviceState* states, int iters,
                                                                              double* sums) {
    const int2 bi = blocks[blockIdx.x];
    const BatchInst I = insts[bi.x];
    FinArgs f = base;
    f.partials = base.partials ? base.partials + I.part_off : nullptr;
    f.grid = I.ctas;
    f.llp = base.llp ? base.llp + I.ll_off : nullptr;
    f.perm = base.perm ? base.perm + I.comp_off : nullptr;
    if (base.masks) {   // point-stationary E-step: per-warp rows, live masks, one ll slot per CTA
        f.masks = base.masks + I.mask_off;
        f.grid = I.ctas * PT_B;
        f.ll_count = I.ctas;
    }
    f.stats64 = base.stats64 ? base.stats64 + (size_t)I.comp_off * NSTAT : nullptr;
    f.shift4 = base.shift4 + I.comp_off;
    f.k = I.k;
    f.n = I.n;
    f.model64 = base.model64 + (size_t)I.comp_off * MODEL;
    f.params = base.params + I.par_off;
    f.trace = base.trace + (size_t)bi.x * iters;
    f.st = states + bi.x;
    reduce_finalize_body(f, bi.y, sums ? sums + (size_t)I.comp_off * NSTAT : nullptr);
}

// The update of every component of a batch, one lane each, from the sums in stats.
__global__ void __launch_bounds__(32) finalize_lanes_batched_kernel(const FinArgs base,
                                                                    const BatchInst* __restrict__ insts,
                                                                    const int* __restrict__ comp_inst, int total_k,
                                                                    DeviceState* states, bool white,
                                                                    const double* __restrict__ stats) {
    const int g = blockIdx.x * 32 + threadIdx.x;
    if (g >= total_k) return;
    const int inst = comp_inst[g];
    const BatchInst I = insts[inst];
    FinArgs f = base;
    f.st = states + inst;
    if ((f.em && f.iter > f.st->stop_after) || f.st->error != 0) return;
    f.perm = base.perm ? base.perm + I.comp_off : nullptr;
    f.shift4 = base.shift4 + I.comp_off;
    f.model64 = base.model64 + (size_t)I.comp_off * MODEL;
    f.params = base.params + I.par_off;
    const int b = g - I.comp_off;
    finalize_update_lane(f, b, white, stats + (size_t)g * NSTAT);
    if (b == 0) f.st->w_raw = 1;
}

// What a given model and its points need before the E-step, in one launch: the first nbuild
// blocks build 32 components each (a binary64 chain per lane, the launch's time) and fill the
// padding slots, the others pack the points meanwhile.  A non-finite point is reported before
// anything wrong with the model, whichever block finds what first.
// Measured: 276,347 points, K = 1023: 7.0 + 2.1 + 5.2 us in three launches, 8.2 us in one.
constexpr int MP_THREADS = 256;
__global__ void __launch_bounds__(MP_THREADS) model_points_kernel(const float* __restrict__ p3, int64_t n,
                                                                  float4* __restrict__ p8,
                                                                  const float* __restrict__ w,
                                                                  const float* __restrict__ mu,
                                                                  const float* __restrict__ cov, int k, int slots,
                                                                  int nbuild, double* model64, float* params,
                                                                  float4* shift4, float4* ctr, float2* aux,
                                                                  DeviceState* st) {
    if ((int)blockIdx.x >= nbuild) {
        const int64_t i = (int64_t)(blockIdx.x - nbuild) * MP_THREADS + threadIdx.x;
        if (i < n && !pack_point(p3, i, nullptr, p8)) atomicExch(&st->error, GIRA_ERR_NONFINITE_INPUT);
        return;
    }
    if (threadIdx.x >= 32) {
        for (int b = k + blockIdx.x * (MP_THREADS - 32) + threadIdx.x - 32; b < slots; b += nbuild * (MP_THREADS - 32))
            pad_slot(params, b);
        return;
    }
    const int b = blockIdx.x * 32 + threadIdx.x;
    float cc = -INFINITY;
    if (b < k) {
        const double pi = w[b];
        const double m[3] = {mu[3 * b], mu[3 * b + 1], mu[3 * b + 2]};
        const float* S = cov + 9 * (size_t)b;
        const double c[6] = {S[0], S[3], S[6], S[4], S[7], S[8]};   // lower triangle, as the oracle reads it
        bool fin = isfinite(pi) && isfinite(m[0]) && isfinite(m[1]) && isfinite(m[2]);
        for (int i = 0; i < 9; ++i) fin = fin && isfinite(S[i]);
        if (!fin) {
            set_error(st, GIRA_ERR_NONFINITE_INPUT);
        } else if (!(pi > 0.0)) {
            set_error(st, GIRA_ERR_INVALID_ARG);
        } else if (build_component(b, pi, m, c, params, shift4, model64, st, b) && ctr) {
            const float* base = params + (size_t)(b >> 1) * PAIR_FLOATS + (b & 1);
            const float s2 = base[2 * SLOT_S];
            cc = base[2 * SLOT_C];
            ctr[b] = make_float4((float)m[0], (float)m[1], (float)m[2], s2);
            aux[b] = f2(cc, s2);
        }
    }
    if (ctr) raise_cmax(st, cc);
}

// ------------------------------------------------------------------ batched helpers
__global__ void params_from_model_batched_kernel(const float* __restrict__ w, const float* __restrict__ mu,
                                                 const float* __restrict__ cov, int total_k,
                                                 const int* __restrict__ comp_inst,
                                                 const BatchInst* __restrict__ insts, double* model64, float* params,
                                                 float4* shift4, DeviceState* states) {
    const int g = blockIdx.x * blockDim.x + threadIdx.x;   // global component
    if (g >= total_k) return;
    const int i = comp_inst[g];
    const BatchInst I = insts[i];
    const int b = g - I.comp_off;
    DeviceState* st = states + i;
    const double pi = w[g];
    const double m[3] = {mu[3 * (size_t)g], mu[3 * (size_t)g + 1], mu[3 * (size_t)g + 2]};
    const float* S = cov + 9 * (size_t)g;
    const double c[6] = {S[0], S[3], S[6], S[4], S[7], S[8]};
    bool fin = isfinite(pi) && isfinite(m[0]) && isfinite(m[1]) && isfinite(m[2]);
    for (int q = 0; q < 9; ++q) fin = fin && isfinite(S[q]);
    if (!fin) { set_error(st, GIRA_ERR_NONFINITE_INPUT); return; }
    if (!(pi > 0.0)) { set_error(st, GIRA_ERR_INVALID_ARG); return; }
    build_component(b, pi, m, c, params + I.par_off, shift4 + I.comp_off, model64 + (size_t)I.comp_off * MODEL, st,
                    b);
}

__global__ void model_out_batched_kernel(const double* __restrict__ model64, const BatchInst* __restrict__ insts,
                                         float* w, float* mu, float* cov, const DeviceState* states,
                                         const int* __restrict__ perm) {
    __shared__ double s_part[2];
    const BatchInst I = insts[blockIdx.x];
    const DeviceState* st = states + blockIdx.x;
    const double* M = model64 + (size_t)I.comp_off * MODEL;
    double part = 0.0;
    for (int a = threadIdx.x; a < I.k; a += blockDim.x) part += M[(size_t)a * MODEL];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) part += __shfl_xor_sync(FULL, part, o);
    if ((threadIdx.x & 31) == 0) s_part[threadIdx.x >> 5] = part;
    __syncthreads();
    const double nsum = s_part[0] + s_part[1];
    if (st->error) return;
    for (int sl = threadIdx.x; sl < I.k; sl += blockDim.x) {   // slot; the caller's index is perm[slot]
        const double* m = M + (size_t)sl * MODEL;
        const size_t g = (size_t)I.comp_off + (perm ? perm[I.comp_off + sl] : sl);
        w[g] = (float)(st->w_raw ? m[0] / nsum : m[0]);
        for (int q = 0; q < 3; ++q) mu[3 * g + q] = (float)m[1 + q];
        const int idx[9] = {0, 1, 2, 1, 3, 4, 2, 4, 5};
        for (int q = 0; q < 9; ++q) cov[9 * g + q] = (float)m[4 + idx[q]];
    }
}

__global__ void model_out_kernel(const double* __restrict__ model64, int k, float* w, float* mu, float* cov,
                                 const DeviceState* st, const int* __restrict__ perm) {
    __shared__ double s_part[2];
    // after an M-step the stored weights are N_b: pi_b = N_b / sum_a N_a (fixed order)
    double part = 0.0;
    for (int a = threadIdx.x; a < k; a += blockDim.x) part += model64[(size_t)a * MODEL];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) part += __shfl_xor_sync(FULL, part, o);
    if ((threadIdx.x & 31) == 0) s_part[threadIdx.x >> 5] = part;
    __syncthreads();
    const double nsum = s_part[0] + s_part[1];
    const int s = blockIdx.x * blockDim.x + threadIdx.x;   // slot; the caller's index is perm[s]
    if (s >= k) return;
    const int b = perm ? perm[s] : s;
    if (!GIRA_IN(b >= 0 && b < k, const_cast<DeviceState*>(st))) return;
    const double* m = model64 + (size_t)s * MODEL;
    w[b] = (float)(st->w_raw ? m[0] / nsum : m[0]);
    for (int i = 0; i < 3; ++i) mu[3 * (size_t)b + i] = (float)m[1 + i];
    const int idx[9] = {0, 1, 2, 1, 3, 4, 2, 4, 5};
    for (int i = 0; i < 9; ++i) cov[9 * (size_t)b + i] = (float)m[4 + idx[i]];
}

// Components in the order of a space-filling curve of their means: the Morton
// code (10 bits per axis over the means' bounding box, binary32) with the index
// as the low bits, sorted by one block (bitonic network in shared memory).
// Slot s then takes the component perm[s]: its row of `old` (a copy of model64)
// is rebuilt into slot s of model64, params and shift4.  Only the order of the
// components in the fit changes: the E-step's per-point sums see them in
// another order, and nothing else.
__device__ __forceinline__ unsigned spread10(unsigned v) {   // bit i -> bit 3 i
    v &= 0x3ffu;
    v = (v | (v << 16)) & 0x030000ffu;
    v = (v | (v << 8)) & 0x0300f00fu;
    v = (v | (v << 4)) & 0x030c30c3u;
    v = (v | (v << 2)) & 0x09249249u;
    return v;
}

// insts (batched fits): block i orders instance i (its own k, offsets and state).
__global__ void __launch_bounds__(ORDER_THREADS) order_components_kernel(const double* __restrict__ old,
                                                                        int stride, int k, int kp2, int* perm,
                                                                        const BatchInst* __restrict__ insts) {
    extern __shared__ unsigned long long keys[];   // kp2 = power of two >= k
    __shared__ float s_lo[3][32], s_hi[3][32];
    if (insts) {
        const BatchInst I = insts[blockIdx.x];
        k = I.k;
        old += (size_t)I.comp_off * stride;
        perm += I.comp_off;
        kp2 = 1;
        while (kp2 < k) kp2 <<= 1;
    }
    const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
    // binary32 (the order only needs coarse cells; rounding to binary32 keeps min and max)
    float lo[3] = {INFINITY, INFINITY, INFINITY}, hi[3] = {-INFINITY, -INFINITY, -INFINITY};
    for (int b = t; b < k; b += blockDim.x)
        for (int i = 0; i < 3; ++i) {
            const float v = (float)old[(size_t)b * stride + 1 + i];
            lo[i] = fminf(lo[i], v);
            hi[i] = fmaxf(hi[i], v);
        }
    for (int i = 0; i < 3; ++i) {
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            lo[i] = fminf(lo[i], __shfl_xor_sync(FULL, lo[i], o));
            hi[i] = fmaxf(hi[i], __shfl_xor_sync(FULL, hi[i], o));
        }
        if (lane == 0) {
            s_lo[i][warp] = lo[i];
            s_hi[i][warp] = hi[i];
        }
    }
    __syncthreads();
    const int nw = blockDim.x >> 5;
    float scale[3];
    for (int i = 0; i < 3; ++i) {
        lo[i] = s_lo[i][0];
        hi[i] = s_hi[i][0];
        for (int w = 1; w < nw; ++w) {
            lo[i] = fminf(lo[i], s_lo[i][w]);
            hi[i] = fmaxf(hi[i], s_hi[i][w]);
        }
        scale[i] = hi[i] > lo[i] ? 1024.f / (hi[i] - lo[i]) : 0.f;
    }
    for (int b = t; b < kp2; b += blockDim.x) {
        unsigned long long key = ~0ull;
        if (b < k) {
            unsigned code = 0;
            for (int i = 0; i < 3; ++i) {
                const float u = ((float)old[(size_t)b * stride + 1 + i] - lo[i]) * scale[i];
                const unsigned q = (unsigned)fminf(1023.f, fmaxf(0.f, floorf(u)));
                code |= spread10(q) << i;
            }
            key = ((unsigned long long)code << 32) | (unsigned)b;
        }
        keys[b] = key;
    }
    __syncthreads();
    for (int size = 2; size <= kp2; size <<= 1)
        for (int hop = size >> 1; hop > 0; hop >>= 1) {
            for (int i = t; i < kp2; i += blockDim.x) {
                const int j = i ^ hop;
                if (j > i) {
                    const unsigned long long a = keys[i], c = keys[j];
                    const bool up = (i & size) == 0;
                    if ((a > c) == up) {
                        keys[i] = c;
                        keys[j] = a;
                    }
                }
            }
            __syncthreads();
        }
    for (int slot = t; slot < k; slot += blockDim.x) perm[slot] = (int)(keys[slot] & 0xffffffffu);
}

// Slot s of every fit takes component perm[s]: its row of `old` rebuilt into slot s
// of model64, params and shift4 (one thread per slot; insts / comp_inst: batched).
__global__ void rebuild_components_kernel(const double* __restrict__ old, const int* __restrict__ perm, int total_k,
                                          double* model64, float* params, float4* shift4, DeviceState* st,
                                          const BatchInst* __restrict__ insts, const int* __restrict__ comp_inst) {
    const int g = blockIdx.x * blockDim.x + threadIdx.x;
    if (g >= total_k) return;
    int slot = g;
    if (insts) {
        const int i = comp_inst[g];
        const BatchInst I = insts[i];
        slot = g - I.comp_off;
        old += (size_t)I.comp_off * MODEL;
        model64 += (size_t)I.comp_off * MODEL;
        params += I.par_off;
        shift4 += I.comp_off;
        st += i;
    }
    const int b = perm[g];
    if (!GIRA_IN(b >= 0 && b < (insts ? insts[comp_inst[g]].k : total_k), st)) return;
    const double* r = old + (size_t)b * MODEL;
    build_component(slot, r[0], r + 1, r + 4, params, shift4, model64, st, b);
}

// ------------------------------------------------------------------ differentiable log-likelihood
// x' = R x + t in binary32 (fixed order), stored as (x,x,y,y)(z,z,0,0).
__global__ void pack_pose_kernel(const float* __restrict__ p3, int64_t n, const float* __restrict__ pose,
                                 float4* __restrict__ p8, DeviceState* st) {
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const float x = p3[3 * i], y = p3[3 * i + 1], z = p3[3 * i + 2];
    float o[3] = {x, y, z};
    if (pose) {
#pragma unroll
        for (int r = 0; r < 3; ++r) o[r] = fmaf(pose[3 * r + 2], z, fmaf(pose[3 * r + 1], y, pose[3 * r] * x)) + pose[9 + r];
    }
    if (!(isfinite(o[0]) && isfinite(o[1]) && isfinite(o[2]))) set_error(st, GIRA_ERR_NONFINITE_INPUT);
    p8[2 * i] = make_float4(o[0], o[0], o[1], o[1]);
    p8[2 * i + 1] = make_float4(o[2], o[2], 0.f, 0.f);
}

// Every point of a batch of scans: x' = R_i x + t_i with the pose of its scan
// (binary search over the offsets); flags non-finite input on its instance.
__global__ void pack_pose_batched_kernel(const float* __restrict__ p3, int64_t n, const int64_t* __restrict__ offsets,
                                         int batch, const float* __restrict__ poses, float4* __restrict__ p8,
                                         DeviceState* states) {
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    int lo = 0, hi = batch;   // offsets[lo] <= i < offsets[hi]
    while (hi - lo > 1) {
        const int mid = (lo + hi) >> 1;
        if (offsets[mid] <= i) lo = mid; else hi = mid;
    }
    const float* pose = poses ? poses + 12 * (size_t)lo : nullptr;
    const float x = p3[3 * i], y = p3[3 * i + 1], z = p3[3 * i + 2];
    float o[3] = {x, y, z};
    if (pose) {
#pragma unroll
        for (int r = 0; r < 3; ++r) o[r] = fmaf(pose[3 * r + 2], z, fmaf(pose[3 * r + 1], y, pose[3 * r] * x)) + pose[9 + r];
    }
    if (!(isfinite(o[0]) && isfinite(o[1]) && isfinite(o[2]))) set_error(states + lo, GIRA_ERR_NONFINITE_INPUT);
    p8[2 * i] = make_float4(o[0], o[0], o[1], o[1]);
    p8[2 * i + 1] = make_float4(o[2], o[2], 0.f, 0.f);
}

// E-step parameters of the gradient from (logits, means, Cholesky factors): pi =
// softmax(logits) in binary64 (max, then fixed-order sums), Sigma_b = L_b L_b^T, then
// the M-step's binary64 build, the components in the order of the Morton code of their
// means (perm[slot] = the caller's component), and their compact arrays for the reach
// tests.  A non-positive diagonal entry of L_b is GIRA_ERR_NOT_PD.
// Bound by the binary64 pipe's latency (a component's build is ~150 dependent warp
// instructions of 64 cycles; K exponentials on one SM take ~6 us), so every block takes
// 32 components, one lane each, and repeats the softmax sums and the Morton ranks
// (each component's rank is the count of smaller keys) instead of waiting for another
// launch.  One block building all K = 1024 took 51 us.  A batch that fills the GPU twice
// that way takes 128 components per block, four warps' lanes: the repeated exponentials
// were its binary64 work (16 models of K = 1024: 41 us with 32, 23 us with 128).
// blockIdx.x: instance (a grid's other dimensions end at 65,535).
constexpr int PFC_THREADS = 256;
template <int PFC_COMPS>   // components built per block
__global__ void __launch_bounds__(PFC_THREADS) params_from_chol_kernel(
    const float* __restrict__ logits, const float* __restrict__ mu, const float* __restrict__ chol, int k,
    const BatchInst* __restrict__ insts, double* model64, float* params, float4* shift4, int* perm, float4* ctr,
    float2* aux, DeviceState* st) {
    __shared__ double s_red[PFC_THREADS / 32];
    __shared__ double s_max, s_lz;
    __shared__ float s_max32[PFC_THREADS / 32];
    __shared__ float s_box[PFC_THREADS / 32][6];
    __shared__ unsigned long long s_key[MAX_K_DIRECT];
    __shared__ int s_slot[PFC_COMPS];
    if (insts) {
        const BatchInst I = insts[blockIdx.x];
        const size_t c = I.comp_off;
        k = I.k;
        logits += c;
        mu += 3 * c;
        chol += 9 * c;
        model64 += c * MODEL;
        params += I.par_off;
        shift4 += c;
        if (perm) {
            perm += c;
            ctr += c;
            aux += c;
        }
        st += blockIdx.x;
    }
    const int c0 = blockIdx.y * PFC_COMPS;
    if (c0 >= k) return;
    const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
    // ---- softmax normaliser, bounding box of the means
    bool fin = true;
    float m = -INFINITY;   // of binary32 values: the binary64 pipe is not needed for it
    float lo[3] = {INFINITY, INFINITY, INFINITY}, hi[3] = {-INFINITY, -INFINITY, -INFINITY};
    for (int b = t; b < k; b += PFC_THREADS) {
        fin = fin && isfinite(logits[b]);
        m = fmaxf(m, logits[b]);
        for (int i = 0; i < 3; ++i) {
            lo[i] = fminf(lo[i], mu[3 * b + i]);
            hi[i] = fmaxf(hi[i], mu[3 * b + i]);
        }
    }
    if (!fin) set_error(st, GIRA_ERR_NONFINITE_INPUT);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        m = fmaxf(m, __shfl_xor_sync(FULL, m, o));
#pragma unroll
        for (int i = 0; i < 3; ++i) {
            lo[i] = fminf(lo[i], __shfl_xor_sync(FULL, lo[i], o));
            hi[i] = fmaxf(hi[i], __shfl_xor_sync(FULL, hi[i], o));
        }
    }
    if (lane == 0) {
        s_max32[warp] = m;
        for (int i = 0; i < 3; ++i) {
            s_box[warp][i] = lo[i];
            s_box[warp][3 + i] = hi[i];
        }
    }
    __syncthreads();
    if (t == 0) {
        float v = s_max32[0];
        for (int w = 1; w < PFC_THREADS / 32; ++w) v = fmaxf(v, s_max32[w]);
        s_max = (double)v;
    }
    float scale[3];
    for (int i = 0; i < 3; ++i) {
        for (int w = 0; w < PFC_THREADS / 32; ++w) {
            lo[i] = fminf(lo[i], s_box[w][i]);
            hi[i] = fmaxf(hi[i], s_box[w][3 + i]);
        }
        scale[i] = hi[i] > lo[i] ? 1024.f / (hi[i] - lo[i]) : 0.f;
    }
    __syncthreads();
    const double amax = s_max;
    double z = 0.0;
    for (int b = t; b < k; b += PFC_THREADS) {
        z += exp((double)logits[b] - amax);
        unsigned code = 0;   // fmaxf / fminf map a NaN to a bound: the keys always give a permutation
        for (int i = 0; i < 3; ++i)
            code |= spread10((unsigned)fminf(1023.f, fmaxf(0.f, floorf((mu[3 * b + i] - lo[i]) * scale[i])))) << i;
        s_key[b] = ((unsigned long long)code << 32) | (unsigned)b;
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) z += __shfl_xor_sync(FULL, z, o);
    __syncthreads();
    if (lane == 0) s_red[warp] = z;
    __syncthreads();
    if (t == 0) {
        double v = 0.0;
        for (int w = 0; w < PFC_THREADS / 32; ++w) v += s_red[w];
        s_lz = amax + log(v);
    }
    // ---- the slots of this block's components: 8 lanes count the smaller keys of each
#pragma unroll
    for (int j0 = 0; j0 < PFC_COMPS; j0 += PFC_THREADS / 8) {
        const int j = j0 + (t >> 3), part = t & 7;
        int cnt = 0;
        if (c0 + j < k) {
            const unsigned long long key = s_key[c0 + j];
            for (int b = part; b < k; b += 8) cnt += s_key[b] < key ? 1 : 0;
        }
#pragma unroll
        for (int o = 4; o > 0; o >>= 1) cnt += __shfl_xor_sync(FULL, cnt, o);
        if (part == 0) s_slot[j] = cnt;
    }
    __syncthreads();
    if (warp >= PFC_COMPS / 32) return;
    const double lz = s_lz;
    const int b = c0 + t;
    float cc = -INFINITY;
    if (b < k) {
        const int slot = perm ? s_slot[t] : b;
        if (perm) perm[slot] = b;
        const float* L = chol + 9 * (size_t)b;
        const double m3[3] = {mu[3 * b], mu[3 * b + 1], mu[3 * b + 2]};
        bool ok = isfinite(m3[0]) && isfinite(m3[1]) && isfinite(m3[2]);
        const double L00 = L[0], L10 = L[3], L11 = L[4], L20 = L[6], L21 = L[7], L22 = L[8];
        ok = ok && isfinite(L00) && isfinite(L10) && isfinite(L11) && isfinite(L20) && isfinite(L21) && isfinite(L22);
        if (!ok) {
            set_error(st, GIRA_ERR_NONFINITE_INPUT);
        } else if (!(L00 > 0.0 && L11 > 0.0 && L22 > 0.0)) {
            atomicMin(&st->bad_component, b);
            set_error(st, GIRA_ERR_NOT_PD);
        } else {
            const double c[6] = {L00 * L00, L00 * L10, L00 * L20, L10 * L10 + L11 * L11, L10 * L20 + L11 * L21,
                                 L20 * L20 + L21 * L21 + L22 * L22};
            if (build_component(slot, exp((double)logits[b] - lz), m3, c, params, shift4, model64, st, b)) {
                const float* base = params + (size_t)(slot >> 1) * PAIR_FLOATS + (slot & 1);
                cc = base[2 * SLOT_C];
                const float s2 = base[2 * SLOT_S];
                if (perm) {
                    ctr[slot] = make_float4((float)m3[0], (float)m3[1], (float)m3[2], s2);
                    aux[slot] = f2(cc, s2);
                }
            }
        }
    }
    raise_cmax(st, cc);
    if (c0 == 0 && (k & 1) && t < PAIR_FLOATS / 2) {   // the odd pair's padding component
        float* base = params + (size_t)(k >> 1) * PAIR_FLOATS + 1;
        base[2 * lane] = lane == SLOT_C ? -INFINITY : 0.f;
    }
}

}  // namespace

cudaError_t launch_reduce_finalize(const float* partials, int grid, const double* ll_partials,
                                   const double* stats64, float4* shift4, int k, int64_t n, double reg, double tol,
                                   double* model64, float* params, double* trace, DeviceState* st, int iter, bool em,
                                   cudaStream_t s, bool pdl, const int* perm, const uint32_t* masks, int nwords,
                                   int ll_count, const uint8_t* cta_key, int* cta_perm, int cta_grid) {
    FinArgs f{partials, grid, ll_partials, stats64, shift4, k, n, reg, tol, model64, params, trace, st, iter,
              em ? 1 : 0, ll_count, 1, perm, masks, nwords};
    const bool order = em && cta_key && cta_perm && cta_grid > 0;
    if (order) {
        f.cta_key = cta_key;
        f.cta_perm = cta_perm;
        f.cta_grid = cta_grid;
    }
    PdlConfig c(dim3((k + FIN_CPB - 1) / FIN_CPB + (order ? 1 : 0)), dim3(FIN_THREADS), 0, s, pdl);
    return cudaLaunchKernelEx(&c.cfg, reduce_finalize_kernel, f);
}

int fin_components_per_block() { return FIN_CPB; }

// Where the binary64 update is the launch (two components of it at a time per block, about
// 1.8 us of an SM's binary64 pipe each), the sums are one launch and the updates, a lane per
// component, another; below eight blocks per SM the update's chain counts and one launch does both.
// 48 segments, 9,488 components: 101 us in one launch, 58 + 11 us in two.
bool finalize_batched_splits(int nblocks) { return nblocks >= 8 * 152; }

cudaError_t launch_reduce_finalize_batched(const float* partials, const double* ll_partials, double* stats64,
                                           float4* shift4, const BatchInst* insts, const int2* blocks, int nblocks,
                                           const int* comp_inst, int total_k, double reg, double tol, int iters,
                                           double* model64, float* params, double* trace, DeviceState* states,
                                           int iter, bool em, cudaStream_t s, const int* perm,
                                           const uint32_t* masks) {
    const bool split = finalize_batched_splits(nblocks);
    const FinArgs f{partials, 0, ll_partials, partials ? nullptr : stats64, shift4, 0, 0, reg, tol, model64, params,
                    trace, nullptr, iter, em ? 1 : 0, 0, 1, perm, masks, 0};
    if (!split || partials)
        reduce_finalize_batched_kernel<<<nblocks, FIN_THREADS, 0, s>>>(f, insts, blocks, states, std::max(iters, 1),
                                                                       split ? stats64 : nullptr);
    if (split)
        finalize_lanes_batched_kernel<<<(total_k + 31) / 32, 32, 0, s>>>(f, insts, comp_inst, total_k, states,
                                                                        partials != nullptr, stats64);
    return cudaGetLastError();
}

cudaError_t launch_fill_padding_batched(float* params, const BatchInst* insts, int batch, int npairs_max,
                                        const int* npairs_of, cudaStream_t s) {
    fill_padding_batched_kernel<<<batch, 128, 0, s>>>(params, insts, npairs_of);
    return cudaGetLastError();
}

cudaError_t launch_params_from_model_batched(const float* w, const float* mu, const float* cov, int total_k,
                                             const int* comp_inst, const BatchInst* insts, double* model64,
                                             float* params, float4* shift4, DeviceState* states, cudaStream_t s) {
    params_from_model_batched_kernel<<<(total_k + 63) / 64, 64, 0, s>>>(w, mu, cov, total_k, comp_inst, insts, model64,
                                                                       params, shift4, states);
    return cudaGetLastError();
}

cudaError_t launch_model_out_batched(const double* model64, const BatchInst* insts, int batch, float* w, float* mu,
                                     float* cov, const DeviceState* states, cudaStream_t s, const int* perm) {
    model_out_batched_kernel<<<batch, 64, 0, s>>>(model64, insts, w, mu, cov, states, perm);
    return cudaGetLastError();
}

cudaError_t launch_ll_reduce_batched(const double* ll_partials, const BatchInst* insts, int batch,
                                     DeviceState* states, cudaStream_t s) {
    ll_reduce_batched_kernel<<<batch, LLR_THREADS, 0, s>>>(ll_partials, insts, states);
    return cudaGetLastError();
}

cudaError_t launch_model_points(const float* pts3, int64_t n, float4* pts8, const float* w, const float* mu,
                                const float* cov, int k, int npairs_pad, double* model64, float* params,
                                float4* shift4, float4* ctr, float2* aux, DeviceState* st, cudaStream_t s) {
    const int nbuild = (k + 31) / 32;
    model_points_kernel<<<(unsigned)(nbuild + (n + MP_THREADS - 1) / MP_THREADS), MP_THREADS, 0, s>>>(
        pts3, n, pts8, w, mu, cov, k, 2 * npairs_pad, nbuild, model64, params, shift4, ctr, aux, st);
    return cudaGetLastError();
}

cudaError_t launch_model_out(const double* model64, int k, float* w, float* mu, float* cov, const DeviceState* st,
                             cudaStream_t s, const int* perm) {
    model_out_kernel<<<(k + 63) / 64, 64, 0, s>>>(model64, k, w, mu, cov, st, perm);
    return cudaGetLastError();
}

cudaError_t launch_order_means(const double* old, int stride, int k, int* perm, cudaStream_t s) {
    if (k > ORDER_MAX_K) return cudaErrorInvalidValue;
    int kp2 = 1;
    while (kp2 < k) kp2 <<= 1;
    const size_t smem = sizeof(unsigned long long) * (size_t)kp2;
    const cudaError_t e =
        cudaFuncSetAttribute(order_components_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    order_components_kernel<<<1, ORDER_THREADS, smem, s>>>(old, stride, k, kp2, perm, nullptr);
    return cudaGetLastError();
}

cudaError_t launch_order_components(double* model64, double* scratch, int k, int* perm, float* params,
                                    float4* shift4, DeviceState* st, cudaStream_t s) {
    if (k > ORDER_MAX_K) return cudaErrorInvalidValue;
    cudaError_t e = cudaMemcpyAsync(scratch, model64, sizeof(double) * (size_t)k * MODEL, cudaMemcpyDeviceToDevice, s);
    if (e != cudaSuccess) return e;
    e = launch_order_means(scratch, MODEL, k, perm, s);
    if (e != cudaSuccess) return e;
    rebuild_components_kernel<<<(k + 63) / 64, 64, 0, s>>>(scratch, perm, k, model64, params, shift4, st, nullptr,
                                                           nullptr);
    return cudaGetLastError();
}

cudaError_t launch_order_components_batched(double* model64, double* scratch, int total_k, int kmax,
                                            const BatchInst* insts, int batch, const int* comp_inst, int* perm,
                                            float* params, float4* shift4, DeviceState* states, cudaStream_t s) {
    if (kmax > ORDER_MAX_K) return cudaErrorInvalidValue;
    cudaError_t e =
        cudaMemcpyAsync(scratch, model64, sizeof(double) * (size_t)total_k * MODEL, cudaMemcpyDeviceToDevice, s);
    if (e != cudaSuccess) return e;
    int kp2 = 1;
    while (kp2 < kmax) kp2 <<= 1;
    const size_t smem = sizeof(unsigned long long) * (size_t)kp2;
    e = cudaFuncSetAttribute(order_components_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    order_components_kernel<<<batch, ORDER_THREADS, smem, s>>>(scratch, MODEL, 0, 0, perm, insts);
    rebuild_components_kernel<<<(total_k + 63) / 64, 64, 0, s>>>(scratch, perm, total_k, model64, params, shift4,
                                                                 states, insts, comp_inst);
    return cudaGetLastError();
}

}  // namespace gira

namespace gira {
cudaError_t launch_pack_pose(const float* pts3, int64_t n, const float* pose12, float4* pts8, DeviceState* st,
                             cudaStream_t s) {
    pack_pose_kernel<<<(unsigned)((n + 255) / 256), 256, 0, s>>>(pts3, n, pose12, pts8, st);
    return cudaGetLastError();
}

cudaError_t launch_params_from_chol(const float* logits, const float* mu, const float* chol, int kmax,
                                    const BatchInst* insts, int batch, double* model64, float* params, float4* shift4,
                                    int* perm, float4* ctr, float2* aux, DeviceState* st, cudaStream_t s) {
    const int nb = insts ? batch : 1;
    if ((int64_t)((kmax + 31) / 32) * nb > 2 * 152) {
        const dim3 grid(nb, (kmax + 127) / 128);
        params_from_chol_kernel<128><<<grid, PFC_THREADS, 0, s>>>(logits, mu, chol, kmax, insts, model64, params,
                                                                  shift4, perm, ctr, aux, st);
    } else {
        const dim3 grid(nb, (kmax + 31) / 32);
        params_from_chol_kernel<32><<<grid, PFC_THREADS, 0, s>>>(logits, mu, chol, kmax, insts, model64, params,
                                                                 shift4, perm, ctr, aux, st);
    }
    return cudaGetLastError();
}

cudaError_t launch_pack_pose_batched(const float* pts3, int64_t n, const int64_t* offsets, int batch,
                                     const float* poses, float4* pts8, DeviceState* states, cudaStream_t s) {
    pack_pose_batched_kernel<<<(unsigned)((n + 255) / 256), 256, 0, s>>>(pts3, n, offsets, batch, poses, pts8,
                                                                         states);
    return cudaGetLastError();
}

}  // namespace gira
