// reach_kernels.cu -- the E-step over many components (3-D with K above 1024, the
// gradient, 4-D): per-block reach lists read from global memory, and the M-step
// statistics accumulated component by component over the blocks each one reaches.
//
// GIRA (arXiv 2307.00071) Sec. V: Eq. (estep) in the log domain (Eq. logestep)
// with the Cholesky log-density of Eq. (simplifiedGaussian).  ex2.approx.ftz
// returns +0 below 2^-126, so a (point, component) whose q' = |P'(x - mu)|^2 +
// (cmax - c) exceeds 126 adds exactly nothing; at thousands of components that is
// all but one pair in fifty or a hundred.
//
// Three kernels per E-step:
//  reach_prepare_kernel  per component (mean, bound of sigma_min(P')^2, c) in compact
//      arrays, and the reference cmax with the weight normaliser;
//  reach_estep_kernel    a block of 128 consecutive points (4 per lane) shared by H
//      warps.  Two tests list the pairs of components that can reach the block: the
//      whole CTA tests every component's sphere against the CTA's box (16 + 8 bytes
//      per component, coalesced), then each warp tests the survivors' boxes exactly as
//      estep_pt_kernel does.  The listed pairs' parameters are read through L1 / L2 as
//      broadcasts: nothing is staged, so shared memory (a few KB of lists) does not
//      bound the occupancy and K does not bound the kernel.  Writes per-point
//      (shift, 1 / total), the log-likelihood, and per block the mask of live pairs;
//  reach_stats_kernel    one warp at a time per (pair, slice of blocks): the statistics of both
//      components over the live blocks of the slice stay in registers and are reduced
//      over the lanes once per slice.  A row-wise second phase would reduce and store 20
//      values per (block, pair) and need a partial row per block (10 GB at 4M points,
//      K = 8192); here it is one 80-byte row per (pair, slice).
// The mode for gradients adds, in reach_estep_kernel, sum_b gamma Sigma_b^-1 (x' - mu_b)
// per point from the live pairs, and the pose sums.
//
// The lists want neighbours in a block: fits and gradients sort the points, the log-likelihood
// takes them as they come (a sensor's order keeps neighbours together; sorting is 60-100 us).
// In no order every pair is listed and the lists are overhead; per call (276,348 points) in
// sensor order and shuffled: K = 2048 199 and 387 us, K = 8192 501 and 1,443; 4-D, K = 512 149
// and 199, K = 2048 282 and 538.  Dense kernels took 465, 1,477, 214 and 550 us in any order.
// Measured on GB300 (4M points of 16 posed frames, K = 8192): E-step 0.72 ms, statistics
// 0.50 ms per iteration; the dense two-pass kernels over chunks of 512 components that
// this replaced took 2 x 15.5 ms.  A call of two iterations with the final
// log-likelihood: 79.2 -> 3.9 ms.
#include <float.h>
#include <math.h>

#include <algorithm>

#include "gira_internal.cuh"

namespace gira {
namespace {

constexpr unsigned FULL = 0xffffffffu;
constexpr float LN2F = 0.693147180559945309f;
constexpr double LN2 = 0.693147180559945309417232121458;
constexpr int RB_P = 4;                    // points per lane
constexpr int RB_PTS = 32 * RB_P;          // points per block (a row of the masks)
constexpr int RB_W = 4;                    // warps per CTA, or those of one block where they are more
__host__ __device__ constexpr int cta_warps(int h) { return h > RB_W ? h : RB_W; }
constexpr float REACH = 128.f;             // q' above which a component is out of reach (e = 0 from q' > 126)

template <int D>
struct Lay;
template <>
struct Lay<3> {
    static constexpr int NP = 6, NS = NSTAT, PF = PAIR_FLOATS;
    static constexpr int SP = SLOT_P, SC = SLOT_C, SNMU = SLOT_NMU, SW = SLOT_W, SS = SLOT_S;
};

template <>
struct Lay<4> {
    static constexpr int NP = 10, NS = NSTAT4, PF = PAIR4_FLOATS;
    static constexpr int SP = SLOT4_P, SC = SLOT4_C, SNMU = SLOT4_NMU, SW = SLOT4_W, SS = SLOT4_S;
};

// Parameters of a pair of components (slot-wise float2: components 2p, 2p + 1).
template <int D>
struct Pair {
    float2 p[Lay<D>::NP], c, nmu[D];
};

// The slots [S0, S0 + N) of pair pp, read as whole float4.
template <int D>
__device__ __forceinline__ void load_slots(const float* params, int pp, float2 (&s)[Lay<D>::PF / 2]) {
    const float4* q = reinterpret_cast<const float4*>(params + (size_t)pp * Lay<D>::PF);
#pragma unroll
    for (int i = 0; i < Lay<D>::PF / 4; ++i) {
        const float4 v = __ldg(q + i);   // slots never used are never loaded (dead after inlining)
        s[2 * i] = f2(v.x, v.y);
        s[2 * i + 1] = f2(v.z, v.w);
    }
}

template <int D>
__device__ __forceinline__ void load_pair(const float* params, int pp, float cmax, Pair<D>& P) {
    float2 s[Lay<D>::PF / 2];
    load_slots<D>(params, pp, s);
#pragma unroll
    for (int i = 0; i < Lay<D>::NP; ++i) P.p[i] = s[Lay<D>::SP + i];
    P.c = f2(cmax - s[Lay<D>::SC].x, cmax - s[Lay<D>::SC].y);
#pragma unroll
    for (int i = 0; i < D; ++i) P.nmu[i] = s[Lay<D>::SNMU + i];
}

// q' = |P'(x - mu)|^2 + (cmax - c) of both components at one point, and y = P'(x - mu)
// (the difference first: see neg_logit2 in em_kernels.cu).
template <int D>
__device__ __forceinline__ float2 nlogit(const Pair<D>& P, const float2 (&X)[D], float2 (&y)[D]) {
    float2 d[D];
#pragma unroll
    for (int j = 0; j < D; ++j) d[j] = add2(X[j], P.nmu[j]);
    float2 q = P.c;
#pragma unroll
    for (int i = 0; i < D; ++i) {
        const int r = i * (i + 1) / 2;
        y[i] = mul2(P.p[r], d[0]);
#pragma unroll
        for (int j = 1; j <= i; ++j) y[i] = fma2(P.p[r + j], d[j], y[i]);
        q = fma2(y[i], y[i], q);
    }
    return q;
}

// max_b c_b: of the prepared references, or (gradient) of the parameter build's atomics
__device__ __forceinline__ float cmax_of(const float* gref, const DeviceState* st) {
    if (gref) return gref[0];
    const int o = st->cmax_ord;
    return __int_as_float(o >= 0 ? o : o ^ 0x7fffffff);
}

template <int D>
__device__ __forceinline__ void load_point(const float4* pts8, int64_t i, float2 (&X)[D]) {
    const float4 a = pts8[2 * i], b = pts8[2 * i + 1];
    X[0] = f2(a.x, a.y);
    X[1] = f2(a.z, a.w);
    X[2] = f2(b.x, b.y);
    if (D == 4) X[D - 1] = f2(b.z, b.w);
}

// ------------------------------------------------------------------ per-component compact arrays
// One block.  ctr[b] = the
// mean's first three coordinates and, in 3-D, the bound s2 of sigma_min(P')^2 (in 4-D the
// fourth coordinate); aux[b] = (c, s2); gref[0] = max_b c_b, gref[1] = the log-likelihood
// reference (cmax - log2 sum_a N_a once the weights are raw N_b, else cmax).
constexpr int PREP_THREADS = 1024;
template <int D>
__global__ void __launch_bounds__(PREP_THREADS) reach_prepare_kernel(const float* __restrict__ params, int k,
                                                                     const DeviceState* st, int iter, float4* ctr,
                                                                     float2* aux, float* gref) {
    __shared__ float s_m[PREP_THREADS / 32];
    __shared__ double s_w[PREP_THREADS / 32];
    pdl_wait();
    if (iter > st->stop_after || st->error) return;
    float m = -INFINITY;
    double w = 0.0;
    for (int b = threadIdx.x; b < k; b += blockDim.x) {
        const float* p = params + (size_t)(b >> 1) * Lay<D>::PF + (b & 1);
        const float c = p[2 * Lay<D>::SC], s2 = p[2 * Lay<D>::SS];
        float x[4];
#pragma unroll
        for (int j = 0; j < D; ++j) x[j] = -p[2 * (Lay<D>::SNMU + j)];
        if (D == 3) x[3] = s2;
        ctr[b] = make_float4(x[0], x[1], x[2], x[3]);
        aux[b] = f2(c, s2);
        m = fmaxf(m, c);
        w += (double)p[2 * Lay<D>::SW];
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        m = fmaxf(m, __shfl_xor_sync(FULL, m, o));
        w += __shfl_xor_sync(FULL, w, o);
    }
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    if (lane == 0) {
        s_m[warp] = m;
        s_w[warp] = w;
    }
    __syncthreads();
    if (warp == 0) {
        m = lane < (int)(blockDim.x >> 5) ? s_m[lane] : -INFINITY;
        w = lane < (int)(blockDim.x >> 5) ? s_w[lane] : 0.0;
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            m = fmaxf(m, __shfl_xor_sync(FULL, m, o));
            w += __shfl_xor_sync(FULL, w, o);
        }
        if (lane == 0) {
            gref[0] = m;
            gref[1] = st->w_raw ? (float)((double)m - log2(w)) : m;
        }
    }
}

// Whether a component of the pair with slots s can have q' <= limit at a point of the box
// (centre ctr, half-extents h): the two lower bounds of estep_pt_kernel's phase 0,
//   |P'(x - mu)| >= |P'(ctr - mu)| - sum_j h_j |column j of P'|  and
//   |P'(x - mu)|^2 >= sigma_min(P')^2 dist(mu, box)^2,
// with their relative slack.  ub (if not nullptr): lowered to the pair's upper bound of
// q' over the box.
template <int D>
__device__ __forceinline__ bool pair_reaches(const float2 (&s)[Lay<D>::PF / 2], const float (&ctr)[D],
                                             const float (&h)[D], float cmax, float limit, float* ub) {
    bool live = false;
#pragma unroll
    for (int m = 0; m < 2; ++m) {
        auto sl = [&](int q) { return m ? s[q].y : s[q].x; };
        const float cc = cmax - sl(Lay<D>::SC), room = limit - cc;   // q' budget left for |y|^2
        float d[D], yy = 0.f, r = 0.f, e2 = 0.f;
#pragma unroll
        for (int j = 0; j < D; ++j) {
            d[j] = ctr[j] + sl(Lay<D>::SNMU + j);
            const float e = fmaxf(fabsf(d[j]) - h[j], 0.f);
            e2 = fmaf(e, e, e2);
            float col = 0.f;   // |column j of P'|^2
#pragma unroll
            for (int i = j; i < D; ++i) {
                const float v = sl(Lay<D>::SP + i * (i + 1) / 2 + j);
                col = fmaf(v, v, col);
            }
            r = fmaf(h[j], sqrtf(col), r);
        }
#pragma unroll
        for (int i = 0; i < D; ++i) {
            float y = 0.f;
#pragma unroll
            for (int j = 0; j <= i; ++j) y = fmaf(sl(Lay<D>::SP + i * (i + 1) / 2 + j), d[j], y);
            yy = fmaf(y, y, yy);
        }
        const float reach = (r + sqrtf(fmaxf(room, 0.f))) * (1.f + 1.f / 256.f);
        const float iso = sl(Lay<D>::SS) * e2 * (1.f - 1.f / 128.f);
        live = live || (room > 0.f && yy <= reach * reach && iso <= room);
        if (ub) {
            const float u = (r + sqrtf(yy)) * (1.f + 1.f / 256.f);
            *ub = fminf(*ub, fmaf(u, u, cc));
        }
    }
    return live;
}

// ------------------------------------------------------------------ the E-step
// Shared memory: the CTA's surviving pairs by warp and class (pp % H), every
// warp's listed pairs, every warp's live-mask words.
__host__ __device__ constexpr int reach_pairs(int k, int h) {   // as many whole warps of pairs as the CTA has warps
    const int step = 32 * cta_warps(h);
    return ((k + 1) / 2 + step - 1) / step * step;
}
__host__ __device__ constexpr int reach_words(int k) { return (((k + 1) / 2) + 31) / 32; }
__host__ __device__ constexpr size_t reach_smem(int k, int h) {
    return (size_t)reach_pairs(k, h) * 2 + (size_t)cta_warps(h) * (reach_pairs(k, h) / h) * 2 +
           (size_t)cta_warps(h) * reach_words(k) * 4;
}

// The barrier of block blk's H warps.
template <int H>
__device__ __forceinline__ void block_sync(int blk) {
    if (H >= RB_W) {
        __syncthreads();
    } else if (blk == 0) {
        asm volatile("bar.sync 1, %0;" ::"n"(32 * H) : "memory");
    } else {
        asm volatile("bar.sync 2, %0;" ::"n"(32 * H) : "memory");
    }
}

// Registers: 3-D without the gradient fits 96 a thread (5 CTAs per SM: the 4M-point map's
// call 3.90 ms, 4.04 with 4); the others would spill (4-D 5.04 against 4.95 ms per frame fit,
// 16 registrations 763 against 698 us).
// MODE 0: log-likelihood; 1: also (shift, 1 / total) and the masks for reach_stats_kernel;
// 2: the gradient (the masks only when a.masks).  H warps share a block's pairs (pp % H):
// 2 for large inputs, 4 where 256-point CTAs would leave SMs idle, 8 or 16 for the
// log-likelihood of few blocks (launch_estep_reach).
template <int D, int H, int MODE>
__global__ void __launch_bounds__(32 * cta_warps(H), H > RB_W ? 16 / H : D == 3 && MODE != 2 ? 5 : 4)
    estep_reach_kernel(const ReachLaunch a_in) {
    extern __shared__ __align__(16) unsigned char dsm[];
    constexpr int W = cta_warps(H), B = W / H;   // warps and blocks per CTA
    static_assert(B * H == W && B <= 2 && (32 % H) == 0, "one named barrier per block, lanes in classes");
    __shared__ float s_box[W][2 * D];
    __shared__ float2 s_tot[W][RB_P][32];
    __shared__ float s_ub[W];
    __shared__ int s_cnt[W][H];
    __shared__ double s_ll[B];
    __shared__ int s_skip;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int blk = warp / H, half = warp % H;
    // batched launches: this CTA's instance.  Everything of the instance is an offset
    // added to the launch's own pointers (loads through a pointer advanced inside a copy
    // of the launch struct read the unadvanced one under nvcc 13.0 for sm_103a).
    int cta = blockIdx.x, inst = 0, k = a_in.k;
    int64_t pt0 = 0, n = a_in.n, rows = a_in.rows, par_off = 0, comp_off = 0, mask_off = 0, ll_off = 0, live_off = 0;
    DeviceState* st = a_in.st;
    if (a_in.units) {
        const BatchUnit u = a_in.units[blockIdx.x];
        const BatchInst I = a_in.insts[u.inst];
        cta = u.cta;
        inst = u.inst;
        pt0 = I.pt_off;
        n = I.n;
        k = I.k;
        rows = (I.n + RB_PTS - 1) / RB_PTS;
        par_off = I.par_off;
        comp_off = I.comp_off;
        mask_off = I.mask_off;
        ll_off = I.ll_off;
        live_off = I.live_off;
        st = a_in.states + u.inst;
    }
    const float* const params = a_in.params + par_off;
    const float4* const ctr4 = a_in.ctr + comp_off;
    const float2* const aux = a_in.aux + comp_off;
    const int npairs = (k + 1) >> 1;
    const int nall = reach_pairs(k, H), nshare = nall / W, ncap = nall / H, nwords = reach_words(k);
    uint16_t* slist0 = reinterpret_cast<uint16_t*>(dsm);          // [W][H][nshare / H]
    uint16_t* slist = slist0 + nall + (size_t)warp * ncap;        // this warp's listed pairs
    uint32_t* smask_all = reinterpret_cast<uint32_t*>(slist0 + nall + (size_t)W * ncap);
    uint32_t* smask = smask_all + warp * nwords;
    // a slot beyond n holds a point 1e18 m away, where every q' is +inf and e exactly 0
    const int64_t row = (int64_t)cta * B + blk;
    const int64_t base = row * RB_PTS + lane;
    float2 X[RB_P][D];
    bool valid[RB_P];
#pragma unroll
    for (int p = 0; p < RB_P; ++p) {
        const int64_t i = base + 32 * p;
        valid[p] = i < n && GIRA_IN(a_in.n_buf == 0 || pt0 + i < a_in.n_buf, st);
        if (valid[p]) {
            load_point<D>(a_in.pts8, pt0 + i, X[p]);
        } else {
#pragma unroll
            for (int j = 0; j < D; ++j) X[p][j] = dup(1e18f);
        }
    }
    float lo[D], hi[D];
#pragma unroll
    for (int j = 0; j < D; ++j) {
        lo[j] = INFINITY;
        hi[j] = -INFINITY;
    }
#pragma unroll
    for (int p = 0; p < RB_P; ++p)
        if (valid[p])
#pragma unroll
            for (int j = 0; j < D; ++j) {
                lo[j] = fminf(lo[j], X[p][j].x);
                hi[j] = fmaxf(hi[j], X[p][j].x);
            }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1)
#pragma unroll
        for (int j = 0; j < D; ++j) {
            lo[j] = fminf(lo[j], __shfl_xor_sync(FULL, lo[j], o));
            hi[j] = fmaxf(hi[j], __shfl_xor_sync(FULL, hi[j], o));
        }
    if (lane == 0)
#pragma unroll
        for (int j = 0; j < D; ++j) {
            s_box[warp][j] = lo[j];
            s_box[warp][D + j] = hi[j];
        }
    pdl_wait();   // the parameters and the state written by the previous kernels
    if (threadIdx.x == 0) s_skip = (a_in.iter > st->stop_after) || (st->error != 0);
    __syncthreads();
    if (s_skip) return;
    pdl_allow_next();
    const float cmax = cmax_of(a_in.gref, st), ref0 = a_in.gref ? a_in.gref[1] : cmax;

    // ---- the components whose sphere {x : sigma_min(P')^2 |x - mu|^2 <= room} meets the
    // CTA's box: a superset of those the second test keeps (a larger box, more slack)
    {
        float blo[D], bhi[D];
#pragma unroll
        for (int j = 0; j < D; ++j) {
            blo[j] = s_box[0][j];
            bhi[j] = s_box[0][D + j];
            if (B == 2) {
                blo[j] = fminf(blo[j], s_box[H][j]);
                bhi[j] = fmaxf(bhi[j], s_box[H][D + j]);
            }
        }
        int cnt = 0;   // lanes of class c keep the count of their class: lane % H == pp % H
        const uint32_t cls = (H == 2 ? 0x55555555u : H == 4 ? 0x11111111u : H == 8 ? 0x01010101u : 0x00010001u) << (lane % H);
        uint16_t* dst = slist0 + warp * nshare + (lane % H) * (nshare / H);
        for (int j0 = 0; j0 < nshare; j0 += 32) {
            const int pp = warp * nshare + j0 + lane;
            bool live = false;
#pragma unroll
            for (int m = 0; m < 2; ++m) {
                const int b = 2 * pp + m;
                if (b < k) {
                    const float4 ct = ctr4[b];
                    const float2 ax = aux[b];
                    const float x[4] = {ct.x, ct.y, ct.z, ct.w};
                    float d2 = 0.f;
#pragma unroll
                    for (int j = 0; j < D; ++j) {
                        const float e = fmaxf(fmaxf(blo[j] - x[j], x[j] - bhi[j]), 0.f);
                        d2 = fmaf(e, e, d2);
                    }
                    const float room = REACH - (cmax - ax.x);
                    live = live || (room > 0.f && ax.y * d2 * (1.f - 1.f / 64.f) <= room);
                }
            }
            const uint32_t m = __ballot_sync(FULL, live) & cls;
            if (live) dst[cnt + __popc(m & ((1u << lane) - 1u))] = (uint16_t)pp;
            cnt += __popc(m);
        }
        if (lane < H) s_cnt[warp][lane] = cnt;
    }
    for (int wd = lane; wd < nwords; wd += 32) smask[wd] = 0u;
    __syncthreads();

    // ---- of these, the pairs of this warp's class that can reach a point of its block
    // (the two bounds of estep_pt_kernel's phase 0, over the block's box)
    int nlive = 0;
    float ctr[D], h[D];
#pragma unroll
    for (int j = 0; j < D; ++j) {
        ctr[j] = 0.5f * (lo[j] + hi[j]);
        h[j] = fmaxf(hi[j] - ctr[j], ctr[j] - lo[j]);
    }
    auto push = [&](bool live, int pp) {   // append the lanes' live pairs in lane order
        const uint32_t m = __ballot_sync(FULL, live);
        const int at = nlive + __popc(m & ((1u << lane) - 1u));
        if (live && GIRA_IN(at < ncap, st)) slist[at] = (uint16_t)pp;
        nlive += __popc(m);
    };
    if (lo[0] <= hi[0]) {
        for (int w = 0; w < W; ++w) {
            const uint16_t* src = slist0 + w * nshare + half * (nshare / H);
            const int cnt = s_cnt[w][half];
            for (int i0 = 0; i0 < cnt; i0 += 32) {
                const int pp = i0 + lane < cnt ? (int)src[i0 + lane] : -1;
                bool live = false;
                if (pp >= 0 && GIRA_IN(pp < npairs, st)) {
                    float2 s[Lay<D>::PF / 2];
                    load_slots<D>(params, pp, s);
                    live = pair_reaches<D>(s, ctr, h, cmax, REACH, nullptr);
                }
                push(live, pp);
            }
        }
    }
    __syncwarp();

    // ---- phase 1: the listed pairs at the lane's points; a pair with a nonzero e is live
    float2 tot[RB_P];
#pragma unroll
    for (int p = 0; p < RB_P; ++p) tot[p] = f2(0.f, 0.f);
    constexpr int U = D == 3 ? 2 : 1;   // pairs per step (4-D: one, for registers)
    for (int i = 0; i < nlive; i += U) {
        int pp[U];
        Pair<D> P[U];
        uint32_t nz[U];
#pragma unroll
        for (int u = 0; u < U; ++u) {
            pp[u] = slist[min(i + u, nlive - 1)];
            load_pair<D>(params, pp[u], cmax, P[u]);
            if (i + u >= nlive) P[u].c = dup(INFINITY);   // no such pair: q' = inf, e = 0
            nz[u] = 0u;
        }
#pragma unroll
        for (int p = 0; p < RB_P; ++p) {
            float2 y[D], s = f2(0.f, 0.f);
#pragma unroll
            for (int u = 0; u < U; ++u) {
                const float2 nq = nlogit<D>(P[u], X[p], y);
                const float2 e = f2(ex2_approx(-nq.x), ex2_approx(-nq.y));
                s = u == 0 ? e : add2(s, e);
                if (MODE != 0) nz[u] |= __float_as_uint(e.x) | __float_as_uint(e.y);
            }
            tot[p] = add2(tot[p], s);
        }
        if (MODE != 0) {
#pragma unroll
            for (int u = 0; u < U; ++u) {
                const bool v = __ballot_sync(FULL, nz[u] != 0u) != 0u;
                if (v && lane == 0) smask[pp[u] >> 5] |= 1u << (pp[u] & 31);
            }
        }
    }

    // ---- totals: the block's warps add their sums in the same order
#pragma unroll
    for (int p = 0; p < RB_P; ++p) s_tot[warp][p][lane] = tot[p];
    block_sync<H>(blk);
    float t[RB_P], sh[RB_P];
    uint32_t rare[RB_P];   // lanes whose point p has every component > 100 binades below cmax
    int nrare = 0;
#pragma unroll
    for (int p = 0; p < RB_P; ++p) {
        t[p] = 0.f;
        sh[p] = 0.f;
#pragma unroll
        for (int h = 0; h < H; ++h) {
            const float2 u = s_tot[blk * H + h][p][lane];
            t[p] += u.x + u.y;
        }
        rare[p] = __ballot_sync(FULL, valid[p] && !(t[p] >= 0x1p-100f));
        nrare += __popc(rare[p]);
    }
    // Rare points: the exact maximum (Eq. logestep's max-subtraction), then the sums
    // relative to it; a pair with a nonzero term becomes live.  The listed pairs give every
    // rare point some q' (or, where none is listed, a pair's upper bound over the box): with U
    // the largest of these over the block's rare points, a pair out of reach of q' <= U + 126
    // adds exact zeros to them, so the pairs are listed again with that limit -- in the
    // registration of a scan 10-20 cm off the model about a third of them, where the maximum
    // over all pairs was two passes over every pair.  nrare is the same in the block's warps.
    if (nrare > 0) {
        float mx[RB_P];
        bool mine[RB_P];
#pragma unroll
        for (int p = 0; p < RB_P; ++p) {
            mx[p] = -INFINITY;
            mine[p] = (rare[p] >> lane) & 1u;
        }
        auto max_pass = [&]() {   // max over the list, then over the block's warps
            for (int i = 0; i < nlive; ++i) {
                Pair<D> P;
                load_pair<D>(params, slist[i], cmax, P);
#pragma unroll
                for (int p = 0; p < RB_P; ++p)
                    if (rare[p]) {
                        float2 y[D];
                        const float2 nq = nlogit<D>(P, X[p], y);
                        mx[p] = fmaxf(mx[p], fmaxf(-nq.x, -nq.y));
                    }
            }
            block_sync<H>(blk);   // s_tot has been read
#pragma unroll
            for (int p = 0; p < RB_P; ++p) s_tot[warp][p][lane] = dup(mx[p]);
            block_sync<H>(blk);
#pragma unroll
            for (int p = 0; p < RB_P; ++p)
#pragma unroll
                for (int g = 0; g < H; ++g) mx[p] = fmaxf(mx[p], s_tot[blk * H + g][p][lane].x);
        };
        max_pass();
        float U = 0.f;
#pragma unroll
        for (int p = 0; p < RB_P; ++p)
            if (mine[p]) U = fmaxf(U, -mx[p]);
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) U = fmaxf(U, __shfl_xor_sync(FULL, U, o));
        if (U == INFINITY) {   // some rare point has no listed pair
            float ub = INFINITY;
            for (int pp = half + H * lane; pp < npairs; pp += 32 * H) {
                float2 s[Lay<D>::PF / 2];
                load_slots<D>(params, pp, s);
                pair_reaches<D>(s, ctr, h, cmax, REACH, &ub);
            }
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) ub = fminf(ub, __shfl_xor_sync(FULL, ub, o));
            if (lane == 0) s_ub[warp] = ub;
            block_sync<H>(blk);
            U = s_ub[blk * H];
#pragma unroll
            for (int g = 1; g < H; ++g) U = fminf(U, s_ub[blk * H + g]);
        }
        nlive = 0;
        for (int j0 = 0; j0 < npairs; j0 += 32 * H) {
            const int pp = j0 + H * lane + half;
            bool live = false;
            if (pp < npairs) {
                float2 s[Lay<D>::PF / 2];
                load_slots<D>(params, pp, s);
                // (a limit beyond binary32, or an overflowing bound: every pair)
                live = !(U < 1e30f) || pair_reaches<D>(s, ctr, h, cmax, U + REACH, nullptr);
            }
            push(live, pp);
        }
        __syncwarp();
        max_pass();
#pragma unroll
        for (int p = 0; p < RB_P; ++p) {
            if (mine[p]) sh[p] = mx[p] > -INFINITY ? -mx[p] : 0.f;
            tot[p] = f2(0.f, 0.f);
        }
        for (int i = 0; i < nlive; ++i) {
            const int pp = slist[i];
            Pair<D> P;
            load_pair<D>(params, pp, cmax, P);
            uint32_t nz = 0u;
#pragma unroll
            for (int p = 0; p < RB_P; ++p)
                if (rare[p]) {
                    float2 y[D];
                    const float2 nq = nlogit<D>(P, X[p], y);
                    const float2 e = f2(ex2_approx(sh[p] - nq.x), ex2_approx(sh[p] - nq.y));
                    tot[p] = add2(tot[p], e);
                    if (mine[p]) nz |= __float_as_uint(e.x) | __float_as_uint(e.y);
                }
            if (MODE != 0) {
                const bool v = __ballot_sync(FULL, nz != 0u) != 0u;
                if (v && lane == 0) smask[pp >> 5] |= 1u << (pp & 31);
            }
        }
        block_sync<H>(blk);
#pragma unroll
        for (int p = 0; p < RB_P; ++p) s_tot[warp][p][lane] = tot[p];
        block_sync<H>(blk);
#pragma unroll
        for (int p = 0; p < RB_P; ++p)
            if (mine[p]) {
                t[p] = 0.f;
#pragma unroll
                for (int g = 0; g < H; ++g) {
                    const float2 u = s_tot[blk * H + g][p][lane];
                    t[p] += u.x + u.y;
                }
            }
    }

    // ---- (shift, 1 / total), log-likelihood
    float2 pr[RB_P];
    double ll = 0.0;
#pragma unroll
    for (int p = 0; p < RB_P; ++p) {
        pr[p] = f2(0.f, 0.f);
        if (valid[p]) {
            if (t[p] > 0.f) {
                pr[p] = f2(sh[p], __frcp_rn(t[p]));
                const float lse2 = lg2_approx(t[p]) + ref0 - sh[p];   // log2 sum_b pi_b N(x|b)
                if (half == 0) {
                    ll += (double)lse2;
                    if (MODE == 0 && a_in.per_point) a_in.per_point[pt0 + base + 32 * p] = lse2 * LN2F;
                }
            } else {
                set_error(st, GIRA_ERR_NUMERIC);   // underflows under every component
            }
            if (MODE != 0 && half == 0 && a_in.masks) a_in.pref[pt0 + base + 32 * p] = pr[p];
        }
    }
    if (half == 0) {
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) ll += __shfl_xor_sync(FULL, ll, o);
        if (lane == 0) s_ll[blk] = ll;
    }
    if (MODE != 0) {
        __syncwarp();
        block_sync<H>(blk);   // the block's masks are final
        if (a_in.masks && half == 0 && row < rows) {
            // the block's mask; the slice's, whose bits first set here become units of work
            int sr;
            const int slices = reach_slices(n, &sr), slice = (int)(row / sr);
            for (int w0 = 0; w0 < nwords; w0 += 32) {
                const int wd = w0 + lane;
                uint32_t m = 0u;
                if (wd < nwords) {
#pragma unroll
                    for (int h2 = 0; h2 < H; ++h2) m |= smask_all[(blk * H + h2) * nwords + wd];
                    a_in.masks[mask_off + wd * rows + row] = m;
                }
                uint32_t fresh = m ? m & ~atomicOr(a_in.live2 + live_off + (int64_t)wd * slices + slice, m) : 0u;
                int incl = __popc(fresh);
#pragma unroll
                for (int o = 1; o < 32; o <<= 1) {
                    const int v = __shfl_up_sync(FULL, incl, o);
                    if (lane >= o) incl += v;
                }
                int at = 0;
                if (lane == 31 && incl) at = atomicAdd(a_in.unit_count, incl);
                at = __shfl_sync(FULL, at, 31) + incl - __popc(fresh);
                for (; fresh; fresh &= fresh - 1u, ++at)
                    a_in.stat_units[at] = make_uint2((unsigned)inst, ((unsigned)slice << 16) | (unsigned)(wd * 32 + __ffs(fresh) - 1));
            }
        }
    }
    if constexpr (MODE == 2) {
        // ---- sum_b gamma P'^T P' (x' - mu) over this warp's live pairs (components packed)
        float2 G[RB_P][D];
#pragma unroll
        for (int p = 0; p < RB_P; ++p)
#pragma unroll
            for (int j = 0; j < D; ++j) {
                G[p][j] = f2(0.f, 0.f);
                if (!valid[p]) X[p][j] = f2(0.f, 0.f);   // weight 0 at a finite place
            }
        for (int wd = 0; wd < nwords; ++wd)
            for (uint32_t m = smask[wd]; m; m &= m - 1u) {
                Pair<D> P;
                load_pair<D>(params, wd * 32 + __ffs(m) - 1, cmax, P);
#pragma unroll
                for (int p = 0; p < RB_P; ++p) {
                    float2 y[D];
                    const float2 nq = nlogit<D>(P, X[p], y);
                    const float2 e = f2(ex2_approx(pr[p].x - nq.x), ex2_approx(pr[p].x - nq.y));
                    const float2 g = mul2(e, dup(pr[p].y));   // pr = 0 for invalid points: g = 0
#pragma unroll
                    for (int j = 0; j < D; ++j) {   // z_j = sum_i P'_ij y_i
                        float2 z = mul2(P.p[j * (j + 1) / 2 + j], y[j]);
#pragma unroll
                        for (int i = j + 1; i < D; ++i) z = fma2(P.p[i * (i + 1) / 2 + j], y[i], z);
                        G[p][j] = fma2(g, z, G[p][j]);
                    }
                }
            }
        // the block's warps in order; -(2 ln 2): P'^T P' = Sigma^{-1} log2(e) / 2
        float g3[RB_P][D];
#pragma unroll
        for (int j = 0; j < D; ++j) {
            block_sync<H>(blk);   // s_tot is free
#pragma unroll
            for (int p = 0; p < RB_P; ++p) s_tot[warp][p][lane] = G[p][j];
            block_sync<H>(blk);
#pragma unroll
            for (int p = 0; p < RB_P; ++p) {
                float v = 0.f;
#pragma unroll
                for (int h = 0; h < H; ++h) {
                    const float2 u = s_tot[blk * H + h][p][lane];
                    v += u.x + u.y;
                }
                g3[p][j] = -1.38629436111989061883f * v;
            }
        }
        __shared__ double s_pose[B][12];
        if (half == 0) {
            float tw[12] = {};   // sum g x'^T (row-major), sum g
#pragma unroll
            for (int p = 0; p < RB_P; ++p) {
                if (!valid[p]) continue;
#pragma unroll
                for (int i = 0; i < 3; ++i) {
#pragma unroll
                    for (int j = 0; j < 3; ++j) tw[3 * i + j] = fmaf(g3[p][i], X[p][j].x, tw[3 * i + j]);
                    tw[9 + i] += g3[p][i];
                }
                if (a_in.grad_pts) {
                    const int64_t at = pt0 + base + 32 * p;
                    float* gp = a_in.grad_pts + 3 * (a_in.order ? (int64_t)a_in.order[at] : at);
                    const float* Rm = a_in.rot + 12 * (size_t)inst;
                    gp[0] = fmaf(Rm[6], g3[p][2], fmaf(Rm[3], g3[p][1], Rm[0] * g3[p][0]));
                    gp[1] = fmaf(Rm[7], g3[p][2], fmaf(Rm[4], g3[p][1], Rm[1] * g3[p][0]));
                    gp[2] = fmaf(Rm[8], g3[p][2], fmaf(Rm[5], g3[p][1], Rm[2] * g3[p][0]));
                }
            }
#pragma unroll
            for (int i = 0; i < 12; ++i) {
                double u = (double)tw[i];
#pragma unroll
                for (int o = 16; o > 0; o >>= 1) u += __shfl_xor_sync(FULL, u, o);
                if (lane == 0) s_pose[blk][i] = u;
            }
        }
        __syncthreads();
        if (threadIdx.x < 12) {
            double u = s_pose[0][threadIdx.x];
            if (B == 2) u += s_pose[B - 1][threadIdx.x];
            a_in.pose_partials[(ll_off + cta) * 12 + threadIdx.x] = u;
        }
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        double v = s_ll[0];
        if (B == 2) v += s_ll[B - 1];
        a_in.llp[ll_off + cta] = v * LN2;
    }
}

// ------------------------------------------------------------------ the statistics
// The E-step listed the (slice, pair)s with work; each warp takes the next one (the order in
// which they were listed and taken decides nothing but who does them): S0 = sum r, S1 = sum
// r y, S2 = sum r y y^T with y = P'(x - mu_old) of both components over the points of the
// slice's live blocks, e formed by the E-step's operations (the same bits), reduced over the
// lanes once and written to row `slice` of the partials [slices][pairs][2 NS].
// Bound by the latency of a block's loads and the length of a warp's chain of blocks.
// Measured: one warp per (pair, slice of 32 or 128 blocks), empty ones among them, 51 us per
// launch on the 276,348-point frame in 4-D at K = 512 and 1.33 ms on the 4M-point map at
// K = 8192, with 9 of 16 resident warps active (CTAs of 8 such warps); 38 us and 0.50 ms now.
// Copying a unit's next block to shared memory meanwhile (cp.async) changed nothing.
// WORLD: about d = x - mu_old instead (a fit repeated after whitened sums lost a covariance to
// binary32: see gira_gmm_fit4).
constexpr int ST_W = 4;   // warps per CTA
template <int D, bool WORLD>
__global__ void __launch_bounds__(32 * ST_W) reach_stats_kernel(const ReachLaunch a_in, float* partials) {
    constexpr int NS = Lay<D>::NS;
    const int lane = threadIdx.x & 31;
    pdl_wait();
    const int count = a_in.unit_count[0];
    auto take = [&]() {
        int u = 0;
        if (lane == 0) u = atomicAdd(a_in.unit_count + 1, 1);
        return __shfl_sync(FULL, u, 0);
    };
    for (int u = take(); u < count; u = take()) {
        const uint2 unit = a_in.stat_units[u];
        const int inst = (int)unit.x, slice = (int)(unit.y >> 16), pp = (int)(unit.y & 0xffffu);
        int k = a_in.k;
        int64_t pt0 = 0, n = a_in.n, rows = a_in.rows, par_off = 0, mask_off = 0, part_off = 0;
        const DeviceState* st = a_in.st;
        if (a_in.insts) {   // offsets into the launch's arrays, as in estep_reach_kernel
            const BatchInst I = a_in.insts[inst];
            pt0 = I.pt_off;
            n = I.n;
            k = I.k;
            rows = (I.n + RB_PTS - 1) / RB_PTS;
            par_off = I.par_off;
            mask_off = I.mask_off;
            part_off = I.part_off;
            st = a_in.states + inst;
        }
        const int npairs = (k + 1) >> 1;
        int sr;
        reach_slices(n, &sr);
        const int64_t r0 = (int64_t)slice * sr, r1 = min(rows, r0 + sr);
        const uint32_t* const mw = a_in.masks + mask_off + (int64_t)(pp >> 5) * rows;
        Pair<D> P;
        load_pair<D>(a_in.params + par_off, pp, cmax_of(a_in.gref, st), P);
        float2 S[NS];
#pragma unroll
        for (int s = 0; s < NS; ++s) S[s] = f2(0.f, 0.f);
        for (int64_t rb = r0; rb < r1; rb += 32) {
            uint32_t m = __ballot_sync(FULL, rb + lane < r1 && ((mw[rb + lane] >> (pp & 31)) & 1u));
            for (; m; m &= m - 1u) {
                const int64_t b0 = (rb + __ffs(m) - 1) * RB_PTS + lane;
#pragma unroll
                for (int p = 0; p < RB_P; ++p) {
                    const int64_t i = b0 + 32 * p;
                    const bool ok = i < n;
                    const int64_t at = pt0 + (ok ? i : n - 1);   // an absent point: the last one with weight 0
                    float2 X[D], y[D];
                    load_point<D>(a_in.pts8, at, X);
                    const float2 pr = a_in.pref[at];
                    const float2 nq = nlogit<D>(P, X, y);
                    const float2 e = f2(ex2_approx(pr.x - nq.x), ex2_approx(pr.x - nq.y));
                    const float2 g = mul2(e, dup(ok ? pr.y : 0.f));
                    if (WORLD)
#pragma unroll
                        for (int j = 0; j < D; ++j) y[j] = add2(X[j], P.nmu[j]);
                    S[0] = add2(S[0], g);
#pragma unroll
                    for (int i2 = 0, q = 1 + D; i2 < D; ++i2) {
                        const float2 gy = mul2(g, y[i2]);
                        S[1 + i2] = add2(S[1 + i2], gy);
#pragma unroll
                        for (int j = i2; j < D; ++j, ++q) S[q] = fma2(gy, y[j], S[q]);
                    }
                }
            }
        }
        // lanes 0-15 end with the first component's sums, 16-31 with the second's
        float v[NS];
        const bool hi16 = lane & 16;
#pragma unroll
        for (int s = 0; s < NS; ++s) {
            const float keep = hi16 ? S[s].y : S[s].x, send = hi16 ? S[s].x : S[s].y;
            v[s] = keep + __shfl_xor_sync(FULL, send, 16);
        }
#pragma unroll
        for (int o = 8; o > 0; o >>= 1)
#pragma unroll
            for (int s = 0; s < NS; ++s) v[s] += __shfl_xor_sync(FULL, v[s], o);
        float mine = 0.f;
#pragma unroll
        for (int s = 0; s < NS; ++s)
            if ((lane & 15) == s) mine = v[s];
        if ((lane & 15) < NS && GIRA_IN(pp < npairs, const_cast<DeviceState*>(st))) {
            float* dst = partials + part_off + ((int64_t)slice * npairs + pp) * (2 * NS);
            dst[(hi16 ? NS : 0) + (lane & 15)] = mine;
        }
    }
}

static_assert(reach_smem(GIRA_MAX_K, 2) <= 40 * 1024 && reach_smem(GIRA_MAX_K, 4) <= 40 * 1024 &&
                  reach_smem(GIRA_MAX_K, 8) <= 36 * 1024 && reach_smem(GIRA_MAX_K, 16) <= 28 * 1024 &&
                  GIRA_MAX_K4 <= GIRA_MAX_K,
              "with the static arrays (5, 5, 10 and 19 KB) within the 48 KB a launch has unasked");

template <int D, int H>
const void* reach_fn(int mode) {
    if constexpr (H <= RB_W) {
        if constexpr (D == 3)   // the gradient is 3-D
            if (mode == 2) return (const void*)estep_reach_kernel<D, H, 2>;
        if (mode == 1) return (const void*)estep_reach_kernel<D, H, 1>;
    }
    return (const void*)estep_reach_kernel<D, H, 0>;
}

}  // namespace

// Two warps per block of 128 points (256-point CTAs), or four (128-point CTAs: a block's
// pairs in parallel, twice the CTAs) up to 8 blocks per SM.  Measured, two against four:
// the gradient of 100k points at K = 1024 924 / 905 us per call, a map of 4M points at
// K = 8192 6.1 / 7.0 ms, its first test then being made twice as often.
// The log-likelihood alone of few blocks under many components takes as many warps as an SM's
// registers hold, sixteen for one block or eight for each of two: four warps walk a block's
// thousands of pairs alone.  Per call, shuffled points: 8,192 at K = 8192 337 us with four warps,
// 152 with sixteen; 20,000 at K = 8192 350 and (eight) 263; up to K = 1024 no difference.
constexpr int RB_FEW_BLOCKS = 152, RB_FEW_K = 1024;
int reach_h(int64_t n) { return n > 152 * 8 * RB_PTS ? 2 : 4; }
int reach_points(int h) { return RB_W / h * RB_PTS; }
int reach_grid(int64_t n) {
    const int64_t pts = reach_points(reach_h(n));
    return (int)std::max<int64_t>(1, (n + pts - 1) / pts);
}
int64_t reach_rows(int64_t n) { return (n + RB_PTS - 1) / RB_PTS; }
int reach_mask_words(int k) { return reach_words(k); }

cudaError_t launch_reach_prepare(int d, const float* params, int k, const DeviceState* st, int iter, float4* ctr,
                                 float2* aux, float* gref, cudaStream_t s) {
    const int threads = std::min(PREP_THREADS, (k + 31) / 32 * 32);
    if (d == 3) reach_prepare_kernel<3><<<1, threads, 0, s>>>(params, k, st, iter, ctr, aux, gref);
    else reach_prepare_kernel<4><<<1, threads, 0, s>>>(params, k, st, iter, ctr, aux, gref);
    return cudaGetLastError();
}

cudaError_t launch_estep_reach(int d, const ReachLaunch& a, int mode, int grid, int h, int kmax, cudaStream_t s) {
    const void* fn = d == 3 ? (h == 2 ? reach_fn<3, 2>(mode) : reach_fn<3, 4>(mode))
                            : (h == 2 ? reach_fn<4, 2>(mode) : reach_fn<4, 4>(mode));
    if (mode == 0 && h == 4 && grid <= 2 * RB_FEW_BLOCKS && kmax > RB_FEW_K) {   // one block per CTA, as with four
        h = grid <= RB_FEW_BLOCKS ? 16 : 8;
        fn = d == 3 ? (h == 8 ? reach_fn<3, 8>(0) : reach_fn<3, 16>(0)) : (h == 8 ? reach_fn<4, 8>(0) : reach_fn<4, 16>(0));
    }
    note_estep_kernel(fn);
    void* args[] = {(void*)&a};
    return cudaLaunchKernel(fn, dim3(grid), dim3(32 * cta_warps(h)), args, reach_smem(kmax, h), s);
}

cudaError_t launch_reach_stats(int d, const ReachLaunch& a, bool world, float* partials, cudaStream_t s) {
    int dev = 0, sms = 1;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    const int grid = sms * (d == 3 ? 7 : 5);   // as many warps as fit (72 and 96 registers a thread)
    if (d == 3) reach_stats_kernel<3, false><<<grid, 32 * ST_W, 0, s>>>(a, partials);
    else if (!world) reach_stats_kernel<4, false><<<grid, 32 * ST_W, 0, s>>>(a, partials);
    else reach_stats_kernel<4, true><<<grid, 32 * ST_W, 0, s>>>(a, partials);
    return cudaGetLastError();
}

// ------------------------------------------------------------------ gradient sums
namespace {

// Block j: 16 pairs of components.  Thread t sums value t of the 16 pairs' 320
// contiguous values over the live slices (compensated binary32, in order); then one
// warp maps the statistics of the 32 components to the parameter gradients in binary64,
// one component per lane (a binary64 warp instruction costs the same whatever the
// number of lanes).  With S0, S1 about y = P'_32 (x' - mu) (the binary32 P' of the E-step;
// P'^T P' = Sigma^{-1} log2(e) / 2):
//   dL/dmu_b    = 2 ln 2 P'^T S1
//   dL/dalpha_b = S0 - N pi_b
// (dL/dL_b: adjoint_kernels.cu).  The instance's block 0 also sums the log-likelihood and
// the pose terms.
constexpr int RG_PAIRS = 16, RG_THREADS = RG_PAIRS * 2 * NSTAT;
static_assert(RG_THREADS % 32 == 0, "whole warps");

__global__ void __launch_bounds__(RG_THREADS) reach_grad_finalize_kernel(const ReachGradArgs f_in,
                                                                         const BatchInst* __restrict__ insts) {
    __shared__ double s_stat[2 * RG_PAIRS][NSTAT];
    // the instance's offsets into the launch's arrays (as in estep_reach_kernel)
    const int inst = blockIdx.x;   // (a grid's other dimensions end at 65,535)
    const BatchInst I = insts[inst];
    int sl;
    const int k = I.k, slices = reach_slices(I.n, &sl), ctas = I.ctas;
    const int64_t n = I.n;
    const size_t c_off = I.comp_off, part_off = I.part_off, live_off = I.live_off, ll_off = I.ll_off, par_off = I.par_off;
    DeviceState* const st = f_in.states + inst;
    const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
    const int npairs = (k + 1) >> 1, pair0 = blockIdx.y * RG_PAIRS;
    if (pair0 >= npairs || st->error) return;
    if (f_in.partials) {
        const int pp = pair0 + t / (2 * NSTAT), v = t % (2 * NSTAT);
        float s = 0.f, e = 0.f;
        if (pp < npairs) {
            const uint32_t* lw = f_in.live2 + live_off + (size_t)(pp >> 5) * slices;
            const float* src = f_in.partials + part_off + (size_t)pp * 2 * NSTAT + v;
            const size_t stride = (size_t)npairs * 2 * NSTAT;
            for (int c0 = 0; c0 < slices; c0 += 8) {   // eight loads in flight
                float x[8];
#pragma unroll
                for (int u = 0; u < 8; ++u)
                    x[u] = (c0 + u < slices && ((lw[c0 + u] >> (pp & 31)) & 1u)) ? src[(size_t)(c0 + u) * stride] : 0.f;
#pragma unroll
                for (int u = 0; u < 8; ++u) {   // Knuth's TwoSum
                    const float a = __fadd_rn(s, x[u]), bp = __fsub_rn(a, s);
                    e = __fadd_rn(e, __fadd_rn(__fsub_rn(s, __fsub_rn(a, bp)), __fsub_rn(x[u], bp)));
                    s = a;
                }
            }
        }
        s_stat[2 * (t / (2 * NSTAT)) + v / NSTAT][v % NSTAT] = (double)s + (double)e;
        __syncthreads();
        const int b = 2 * pair0 + lane;   // this lane's component (slot)
        if (warp == 0 && b < k) {
            const double* S = s_stat[lane];
            const int src_b = f_in.perm[c_off + b];
            const float* q = f_in.params + par_off + (size_t)(b >> 1) * PAIR_FLOATS + (b & 1);
#pragma unroll
            for (int i = 0; i < 3; ++i) {
                double gm = 0.0;
#pragma unroll
                for (int m = i; m < 3; ++m) gm += (double)q[2 * (SLOT_P + m * (m + 1) / 2 + i)] * S[1 + m];
                f_in.g_means[3 * (c_off + src_b) + i] = (float)(1.3862943611198906 * gm);
            }
            f_in.g_logits[c_off + src_b] = (float)(S[0] - (double)n * f_in.model64[(c_off + b) * MODEL]);
        }
    }
    if (blockIdx.y != 0 || warp != 1) return;
    // log-likelihood and pose sums, fixed order
    double v[13] = {};
    for (int c = lane; c < ctas; c += 32) {
        v[0] += f_in.llp[ll_off + c];
#pragma unroll
        for (int i = 0; i < 12; ++i) v[1 + i] += f_in.pp[(ll_off + c) * 12 + i];
    }
#pragma unroll
    for (int i = 0; i < 13; ++i) {
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) v[i] += __shfl_xor_sync(FULL, v[i], o);
    }
    if (lane == 0) {
        st->ll_sum = v[0];
        const double* M = v + 1;    // sum g x'^T
        const double* G = v + 10;   // sum g
        {
            double* const g_twist = f_in.g_twist + 6 * (size_t)inst;   // omega = sum x' x g, v = sum g
            g_twist[0] = M[3 * 2 + 1] - M[3 * 1 + 2];
            g_twist[1] = M[3 * 0 + 2] - M[3 * 2 + 0];
            g_twist[2] = M[3 * 1 + 0] - M[3 * 0 + 1];
            for (int i = 0; i < 3; ++i) g_twist[3 + i] = G[i];
        }
        {   // x = R^T (x' - t): dL/dR = (sum g x'^T - G t^T) R, dL/dt = G
            const float* const pose = f_in.poses + 12 * (size_t)inst;
            double* const g_pose = f_in.g_pose + 12 * (size_t)inst;
            const double tt[3] = {pose[9], pose[10], pose[11]};
            for (int i = 0; i < 3; ++i)
                for (int j = 0; j < 3; ++j) {
                    double acc = 0.0;
                    for (int m = 0; m < 3; ++m) acc += (M[3 * i + m] - G[i] * tt[m]) * (double)pose[3 * m + j];
                    g_pose[3 * i + j] = acc;
                }
            for (int i = 0; i < 3; ++i) g_pose[9 + i] = G[i];
        }
    }
}

}  // namespace

// Without parameter gradients one block per instance.
cudaError_t launch_reach_grad_finalize(const ReachGradArgs& f, const BatchInst* insts, int batch, cudaStream_t s) {
    const int blocks = f.partials ? ((f.kmax + 1) / 2 + RG_PAIRS - 1) / RG_PAIRS : 1;
    reach_grad_finalize_kernel<<<dim3(batch, blocks), RG_THREADS, 0, s>>>(f, insts);
    return cudaGetLastError();
}

}  // namespace gira
