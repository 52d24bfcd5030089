// d4_kernels.cu -- the fit in four dimensions (xyz + intensity, the paper's
// SOGMM data), Gaussian-mixture regression of intensity on xyz, and sampling
// from a mixture.
//
// GIRA (arXiv 2307.00071) Sec. V: the E-step of Eq. (estep) in the log domain
// of Eq. (logestep), the log-density of Eq. (simplifiedGaussian) with D = 4
// (the (1,K,4)/(1,K,4,4) layout of the paper's model), the standard M-step on
// the sufficient statistics; Sec. IV's use of the model: intensity inferred at
// given positions (conditional mean and variance) and points resampled from
// the joint distribution.
//
// The E-step and its statistics are reach_kernels.cu with D = 4 (logits from d = x - mu_b:
// intensity and metre-scale coordinates share a point), or, for little work, the dense
// kernel here; also the M-step, KInit's Lloyd iterations and one-hot statistics, the
// regression and the sampling.
#include <float.h>
#include <math.h>

#include <algorithm>

#include "gira_internal.cuh"

namespace gira {

namespace {

constexpr unsigned FULL = 0xffffffffu;
// lower-triangular index of (i, j), j <= i: 00,10,11,20,21,22,30,31,32,33
__host__ __device__ constexpr int tri4(int i, int j) { return i * (i + 1) / 2 + j; }

// Slot s of component b in the pair-interleaved parameter buffer.
__host__ __device__ __forceinline__ size_t slot4(int b, int s) {
    return (size_t)(b >> 1) * PAIR4_FLOATS + 2 * s + (b & 1);
}

constexpr double ALPHA4 = 0.84932180028801904272;     // sqrt(log2(e) / 2)
constexpr double LOG2_2PI4 = 2.6514961294723187980;   // log2(2 pi)

// A lower bound of sigma_min(P')^2 = alpha^2 / lambda_max(Sigma) from the sum of Sigma's
// squared entries: lambda_max <= ||Sigma||_F (and >= half of it).
__device__ __forceinline__ float sigma_min_sq_bound4(double fro2) {
    return (float)(ALPHA4 * ALPHA4) / (sqrtf((float)fro2) * (1.f + 1e-4f)) * (1.f - 1e-4f);
}

// ------------------------------------------------------------------ the E-step of little work
// Every component at every point, statistics in the same pass: the lists of reach_kernels.cu
// (prepare, E-step, statistics over them, one launch each) save nothing where the dense work
// is a few microseconds.  One CTA holds all K <= 1024 components, one pair per lane; all lanes
// walk the CTA's points (staged by one TMA bulk copy) together, eight at a time: pass 1
// forms e and the per-point sums over lanes and warps, pass 2 the statistics about y = P'(x - mu)
// of both components, packed.  Rows [cta][pairs][2 NSTAT4], every one written.
// Bound by the chain of a batch (the sums cross the warps) and, per launch, by latency.
// Measured: 6 us an iteration for 2,000 points at K = 64, where the lists' prepare, E-step and
// statistics take 5, 10 and 16; a call of 20 iterations 1,168 -> 546 us (both sides of the rule
// at estep4_dense).
constexpr int Q4 = 8;                             // points per batch
constexpr int PPC4_MAX = 1024;                    // points staged per CTA (32 KB)
constexpr long long MBAR_LIMIT4 = 2000000000ll;   // bound on the TMA wait: 2 s of wall time
constexpr float LN2F4 = 0.693147180559945309f;
constexpr double LN2_4 = 0.693147180559945309417232121458;

template <bool STATS, bool WORLD = false>   // WORLD: the statistics about x - mu, as in reach_stats_kernel
__global__ void __launch_bounds__(512, 1) estep4_dense_kernel(const EStep4Launch a) {
    extern __shared__ __align__(128) unsigned char dsm4[];
    __shared__ __align__(8) uint64_t bar_tma;
    __shared__ float red_sum[2][16][Q4];   // by parity of the batch: one barrier per batch
    __shared__ float red_aux[2][16][Q4];
    __shared__ float s_cmax[16], s_wsum[16];
    __shared__ int s_skip, s_norm, s_dead;
    constexpr int LPQ = 32 / Q4;
    const int G = blockDim.x >> 5, warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int pr = threadIdx.x, npairs = (a.k + 1) >> 1;   // this lane's pair
    const int64_t begin = (int64_t)blockIdx.x * a.pts_per_cta;
    const int npts = (int)(min(a.n, begin + a.pts_per_cta) - begin);
    const float4* spts = reinterpret_cast<const float4*>(dsm4);   // (x,x,y,y)(z,z,w,w) per point
    if (threadIdx.x == 0) {
        // the points are never written by the kernel this one may overlap
        // (dependent launch), so their copy starts before the wait below
        mbar_init(&bar_tma, 1);
        mbar_fence_init();
        mbar_expect_tx(&bar_tma, (uint32_t)npts * 32u);
        tma_load_1d(reinterpret_cast<void*>(dsm4), a.pts8 + 2 * begin, (uint32_t)npts * 32u, &bar_tma);
    }
    pdl_wait();   // the parameters and the state written by the previous kernel
    if (threadIdx.x == 0) {
        s_skip = (a.iter > a.st->stop_after) || (a.st->error != 0);
        s_norm = a.st->w_raw;
        s_dead = 0;
    }
    __syncthreads();
    if (s_skip) {   // let the copy land before leaving
        if (threadIdx.x == 0) mbar_wait_bounded(&bar_tma, 0u, MBAR_LIMIT4);
        return;
    }
    pdl_allow_next();
    // ---- this lane's pair (lanes beyond the last: c = -inf, never contribute)
    float2 P[10], nmu[4], c = dup(-INFINITY), w = dup(0.f);
#pragma unroll
    for (int i = 0; i < 10; ++i) P[i] = dup(0.f);
#pragma unroll
    for (int i = 0; i < 4; ++i) nmu[i] = dup(0.f);
    if (pr < npairs) {
        const float4* src = reinterpret_cast<const float4*>(a.params + (size_t)pr * PAIR4_FLOATS);
        float4 v[8];
#pragma unroll
        for (int i = 0; i < 8; ++i) v[i] = src[i];
        const float2* f = reinterpret_cast<const float2*>(v);
#pragma unroll
        for (int i = 0; i < 10; ++i) P[i] = f[SLOT4_P + i];
        c = f[SLOT4_C];
#pragma unroll
        for (int i = 0; i < 4; ++i) nmu[i] = f[SLOT4_NMU + i];
        w = f[SLOT4_W];
    }
    float cm = fmaxf(c.x, c.y), ws = w.x + w.y;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        cm = fmaxf(cm, __shfl_xor_sync(FULL, cm, o));
        ws += __shfl_xor_sync(FULL, ws, o);
    }
    if (lane == 0) {
        s_cmax[warp] = cm;
        s_wsum[warp] = ws;
    }
    if (!mbar_wait_bounded(&bar_tma, 0u, MBAR_LIMIT4)) s_dead = 1;
    __syncthreads();
    if (s_dead) {   // the points never arrived: report, let the copy land, leave
        if (threadIdx.x == 0) {
            set_error(a.st, GIRA_ERR_TIMEOUT);
            mbar_wait_bounded(&bar_tma, 0u, MBAR_LIMIT4);
        }
        return;
    }
    float cmax = s_cmax[0], wsum = s_wsum[0];
    for (int i = 1; i < G; ++i) {
        cmax = fmaxf(cmax, s_cmax[i]);
        wsum += s_wsum[i];
    }
    const float2 cc = f2(cmax - c.x, cmax - c.y);   // >= 0; +inf for padding
    const float ref0 = s_norm ? cmax - __log2f(wsum) : cmax;
    float2 S[NSTAT4];
#pragma unroll
    for (int i = 0; i < NSTAT4; ++i) S[i] = f2(0.f, 0.f);
    double ll_acc = 0.0;
    const int myq = q_of_lane<Q4>(lane);
    const bool owner = warp == 0 && (lane & (LPQ - 1)) == 0;
    // y = P'(x - mu) at point li, and q' = |y|^2 + (cmax - c): minus the logit relative to cmax
    auto whiten = [&](int li, float2 (&y)[4]) {
        const float4 xy = spts[2 * li], zw = spts[2 * li + 1];
        const float2 d0 = add2(f2(xy.x, xy.y), nmu[0]), d1 = add2(f2(xy.z, xy.w), nmu[1]);
        const float2 d2 = add2(f2(zw.x, zw.y), nmu[2]), d3 = add2(f2(zw.z, zw.w), nmu[3]);
        y[0] = mul2(P[0], d0);
        y[1] = fma2(P[2], d1, mul2(P[1], d0));
        y[2] = fma2(P[5], d2, fma2(P[4], d1, mul2(P[3], d0)));
        y[3] = fma2(P[9], d3, fma2(P[8], d2, fma2(P[7], d1, mul2(P[6], d0))));
    };
    auto qform = [&](int li) {
        float2 y[4];
        whiten(li, y);
        return fma2(y[3], y[3], fma2(y[2], y[2], fma2(y[1], y[1], fma2(y[0], y[0], cc))));
    };
    float2 E[Q4];
    for (int t = 0, lb = 0; lb < npts; ++t, lb += Q4) {
        const int nvalid = min(Q4, npts - lb);
        float part[Q4];
#pragma unroll
        for (int q = 0; q < Q4; ++q) {
            const float2 nq = qform(q < nvalid ? lb + q : lb);
            E[q] = f2(ex2_approx(-nq.x), ex2_approx(-nq.y));
            part[q] = E[q].x + E[q].y;
        }
        const float wt = warp_transpose_reduce<Q4>(part, lane, AddOp());
        if ((lane & (LPQ - 1)) == 0) red_sum[t & 1][warp][myq] = wt;
        __syncthreads();
        float tot = red_sum[t & 1][0][myq];
        for (int i = 1; i < G; ++i) tot += red_sum[t & 1][i][myq];
        const bool myvalid = myq < nvalid;
        float ref = ref0;
        if (__any_sync(FULL, myvalid && !(tot >= 0x1p-100f))) {
            // rare, the same in every warp: a point > 100 binades below cmax everywhere; the exact
            // per-point maximum
            float m[Q4];
#pragma unroll
            for (int q = 0; q < Q4; ++q) {
                const float2 nq = qform(q < nvalid ? lb + q : lb);
                E[q] = f2(-nq.x, -nq.y);
                m[q] = fmaxf(E[q].x, E[q].y);
            }
            float mt = warp_transpose_reduce<Q4>(m, lane, MaxOp());
            if ((lane & (LPQ - 1)) == 0) red_aux[0][warp][myq] = mt;
            __syncthreads();
            mt = red_aux[0][0][myq];
            for (int i = 1; i < G; ++i) mt = fmaxf(mt, red_aux[0][i][myq]);
            float p2[Q4];
#pragma unroll
            for (int q = 0; q < Q4; ++q) {
                float mq = __shfl_sync(FULL, mt, q * LPQ);
                mq = mq > -INFINITY ? mq : 0.f;
                E[q] = f2(ex2_approx(E[q].x - mq), ex2_approx(E[q].y - mq));
                p2[q] = E[q].x + E[q].y;
            }
            const float w2 = warp_transpose_reduce<Q4>(p2, lane, AddOp());
            if ((lane & (LPQ - 1)) == 0) red_aux[1][warp][myq] = w2;
            __syncthreads();
            tot = red_aux[1][0][myq];
            for (int i = 1; i < G; ++i) tot += red_aux[1][i][myq];
            if (myvalid && !(mt > -INFINITY)) set_error(a.st, GIRA_ERR_NUMERIC);
            ref = ref0 + (mt > -INFINITY ? mt : 0.f);
        }
        const bool ok = myvalid && tot > 0.f;
        const float lse2 = lg2_approx(tot) + ref;
        if (owner && ok) {
            ll_acc += (double)lse2;
            if (!STATS && a.per_point) a.per_point[begin + lb + myq] = lse2 * LN2F4;
        }
        if (STATS) {
            const float r = ok ? __frcp_rn(tot) : 0.f;
#pragma unroll
            for (int q = 0; q < Q4; ++q) {
                const float2 g = mul2(E[q], dup(__shfl_sync(FULL, r, q * LPQ)));
                float2 y[4];
                if (WORLD) {
                    const int li = q < nvalid ? lb + q : lb;
                    const float4 xy = spts[2 * li], zw = spts[2 * li + 1];
                    y[0] = add2(f2(xy.x, xy.y), nmu[0]);
                    y[1] = add2(f2(xy.z, xy.w), nmu[1]);
                    y[2] = add2(f2(zw.x, zw.y), nmu[2]);
                    y[3] = add2(f2(zw.z, zw.w), nmu[3]);
                } else {
                    whiten(q < nvalid ? lb + q : lb, y);
                }
                S[0] = add2(S[0], g);
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    const float2 gy = mul2(g, y[i]);
                    S[1 + i] = add2(S[1 + i], gy);
#pragma unroll
                    for (int j = i; j < 4; ++j) S[5 + sym4(i, j)] = fma2(gy, y[j], S[5 + sym4(i, j)]);
                }
            }
        }
    }
    if (STATS && pr < npairs) {
        float* dst = a.partials + ((size_t)blockIdx.x * npairs + pr) * (2 * NSTAT4);
#pragma unroll
        for (int i = 0; i < NSTAT4; ++i) {
            dst[i] = S[i].x;
            dst[NSTAT4 + i] = S[i].y;
        }
    }
    if (warp == 0) {   // the owner lanes hold the per-point sums; fixed order
#pragma unroll
        for (int o = LPQ; o < 32; o <<= 1) ll_acc += __shfl_xor_sync(FULL, ll_acc, o);
        if (lane == 0) a.ll_partials[blockIdx.x] = ll_acc * LN2_4;
    }
}

// From (w, mu, Sigma) in binary64: Cholesky, P = L^{-1}, the base-2 constants.
// report: the caller's index of the component (slot b may hold another one).
__device__ bool build_component4(int b, double w, const double mu[4], const double S[16], float* params,
                                 double* model64, DeviceState* st, int report) {
    double L[16] = {0};
    bool pd = true;
    for (int j = 0; j < 4 && pd; ++j) {
        double s = S[4 * j + j];
        for (int k = 0; k < j; ++k) s -= L[4 * j + k] * L[4 * j + k];
        if (!(s > 0.0)) { pd = false; break; }
        L[4 * j + j] = sqrt(s);
        for (int i = j + 1; i < 4; ++i) {
            double t = S[4 * i + j];
            for (int k = 0; k < j; ++k) t -= L[4 * i + k] * L[4 * j + k];
            L[4 * i + j] = t / L[4 * j + j];
        }
    }
    if (!pd) {
        atomicMin(&st->bad_component, report);
        set_error(st, GIRA_ERR_NOT_PD);
        return false;
    }
    double P[16] = {0};
    for (int cidx = 0; cidx < 4; ++cidx)
        for (int i = cidx; i < 4; ++i) {
            double t = (i == cidx) ? 1.0 : 0.0;
            for (int k = cidx; k < i; ++k) t -= L[4 * i + k] * P[4 * k + cidx];
            P[4 * i + cidx] = t / L[4 * i + i];
        }
    double fro2 = 0.0;
    for (int i = 0; i < 16; ++i) fro2 += S[i] * S[i];
    params[slot4(b, SLOT4_S)] = sigma_min_sq_bound4(fro2);
    for (int i = 0; i < 4; ++i)
        for (int j = 0; j <= i; ++j) params[slot4(b, SLOT4_P + tri4(i, j))] = (float)(ALPHA4 * P[4 * i + j]);
    // log2 w + sum_j log2 P_jj - (4/2) log2(2 pi)
    params[slot4(b, SLOT4_C)] = (float)(log2(w * (P[0] * P[5] * P[10] * P[15])) - 2.0 * LOG2_2PI4);
    for (int i = 0; i < 4; ++i) params[slot4(b, SLOT4_NMU + i)] = -(float)mu[i];
    params[slot4(b, SLOT4_W)] = (float)w;
    double* m = model64 + (size_t)b * MODEL4;
    m[0] = w;
    for (int i = 0; i < 4; ++i) m[1 + i] = mu[i];
    for (int i = 0; i < 4; ++i)
        for (int j = i; j < 4; ++j) m[5 + sym4(i, j)] = S[4 * i + j];
    return true;
}

// The M-step of one pair of components per block.  Sums: warp w adds, value by lane, the
// pair's live rows among the w-th eighth of the slices (compensated binary32, Knuth's
// TwoSum), warp 0 joins them in order.  Update: warp 0, lanes 16 h + 4 i + j for
// entry (i, j) of component h's 4 x 4 matrices, every stage in parallel lanes through
// shared memory: GB300 issues one binary64 warp instruction per 64 cycles per warp whatever
// the number of active lanes, so a stage costs what one entry costs (~170 instructions in
// all; one thread per component, one block each, ran ~500 in a row: 58 us per launch at
// K = 512, 16 us now under a profiler that empties the caches).  The statistics are about y = P'(x - s) with the binary32 P' of
// the E-step (a component thin in one direction keeps that direction's digits): with M =
// P'^{-1}, mu = (S0 / N_b) s + M ybar, Sigma = M (S2 / N_b - ybar ybar^T) M^T + reg I; one-hot
// statistics are about shift4 with M = I.
struct Fin4Args {
    const float* partials;
    const uint32_t* live2;
    int slices;
    const double* llp;
    int ll_count;
    const double* stats64;
    const float4* shift4;
    int k;
    int64_t n;
    double reg, tol;
    double* model64;
    float* params;
    double* trace;
    const int* perm;
    DeviceState* st;
    int iter, em;
    Sums4 sums;
};
// Binary32 sums whitened by the old components lose part of Sigma = M C M^T on the way back: of Sigma_ii up to
// 2^-24 root_i^2, root_i = sum_m |M_im| (S2_mm / N_b)^(1/2).  One point 1e2 .. 1e6 off in one coordinate of a cloud
// of unit extent: normalised errors of 0.1 .. 2.5 times 2^-24 root_i^2 / Sigma_ii (from 1e-5 to above 1), sums about
// x - mu 2e-6.  From root_i = 16 sqrt(Sigma_ii) on (1.5e-5) the fit goes over to those;
// 256 fits of depth frames (2 .. 15,000 points a component) stayed below 8.1.
constexpr float MAX_LOSS4 = 16.f;
constexpr int FIN4_WARPS = 8;
__global__ void __launch_bounds__(32 * FIN4_WARPS) reduce_finalize4_kernel(const Fin4Args f) {
    __shared__ float s_hi[FIN4_WARPS][2][32];
    __shared__ double s_stat[2][NSTAT4], s_P[2][10], s_r[2][5], s_M[2][16], s_C[2][16], s_A[2][16], s_mu[2][4];
    __shared__ double s_ll[FIN4_WARPS];
    DeviceState* const st = f.st;
    pdl_wait();         // the E-step's partials (dependent launch)
    pdl_allow_next();
    if ((f.em && f.iter > st->stop_after) || st->error) return;
    const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
    const int pp = blockIdx.x;
    const bool white = f.partials != nullptr && f.sums != Sums4::About;
    if (f.partials) {
        const int npairs = (f.k + 1) >> 1;
        const uint32_t* lw = f.live2 ? f.live2 + (size_t)(pp >> 5) * f.slices : nullptr;   // nullptr: every row
        const float* src = f.partials + (size_t)pp * 2 * NSTAT4 + lane;
        const size_t stride = (size_t)npairs * 2 * NSTAT4;
        const int c0 = warp * f.slices / FIN4_WARPS, c1 = (warp + 1) * f.slices / FIN4_WARPS;
        float s = 0.f, e = 0.f;
        auto add = [&](float x) {
            const float a = __fadd_rn(s, x), bp = __fsub_rn(a, s);
            e = __fadd_rn(e, __fadd_rn(__fsub_rn(s, __fsub_rn(a, bp)), __fsub_rn(x, bp)));
            s = a;
        };
        for (int c = c0; c < c1; c += 8) {   // eight loads in flight
            float x[8];
#pragma unroll
            for (int u = 0; u < 8; ++u)
                x[u] = c + u < c1 && lane < 2 * NSTAT4 && (!lw || ((lw[c + u] >> (pp & 31)) & 1u))
                           ? src[(size_t)(c + u) * stride]
                           : 0.f;
#pragma unroll
            for (int u = 0; u < 8; ++u) add(x[u]);
        }
        s_hi[warp][0][lane] = s;
        s_hi[warp][1][lane] = e;
        __syncthreads();
        if (warp == 0) {
#pragma unroll
            for (int w = 1; w < FIN4_WARPS; ++w) {
                e = __fadd_rn(e, s_hi[w][1][lane]);
                add(s_hi[w][0][lane]);
            }
            if (lane < 2 * NSTAT4) s_stat[lane / NSTAT4][lane % NSTAT4] = (double)s + (double)e;
        }
    } else if (warp == 0 && lane < 2 * NSTAT4 && 2 * pp + lane / NSTAT4 < f.k) {
        s_stat[lane / NSTAT4][lane % NSTAT4] = f.stats64[(size_t)2 * pp * NSTAT4 + lane];
    }
    if (warp == 0) {
        const int h = lane >> 4, l = lane & 15, i = l >> 2, j = l & 3;
        const int b = 2 * pp + h;
        const bool on = b < f.k;
        double* P = s_P[h];
        double* r = s_r[h];
        double* M = s_M[h];
        double* C = s_C[h];
        double* A = s_A[h];
        double* mu = s_mu[h];
        const double* S = s_stat[h];
        if (on && l < 10) P[l] = white ? (double)f.params[slot4(b, SLOT4_P + l)] : 0.0;
        __syncwarp();
        const double nbw = on ? S[0] + 10.0 * DBL_EPSILON : 1.0;
        if (on && l < 5) r[l] = __drcp_rn(l == 4 ? nbw : white ? P[tri4(l, l)] : 1.0);
        __syncwarp();
        const double inv = on ? r[4] : 0.0;
        // M = P'^{-1}, row by row (columns in parallel)
        if (on) M[l] = i == j ? r[i] : 0.0;
        __syncwarp();
        if (white)
            for (int row = 1; row < 4; ++row) {
                if (on && i == row && j < row) {
                    double v = 0.0;
                    for (int m = j; m < row; ++m) v = __fma_rn(P[tri4(row, m)], M[4 * m + j], v);
                    M[l] = -v * r[row];
                }
                __syncwarp();
            }
        // C = S2 / N_b - ybar ybar^T
        if (on) C[l] = __fma_rn(-(S[1 + i] * inv), S[1 + j] * inv, S[5 + sym4(min(i, j), max(i, j))] * inv);
        __syncwarp();
        // mu = (S0 / N_b) s + M ybar (lanes 0 .. 3), A = M C
        if (on && l < 4) {
            double s;
            if (f.partials) s = -(double)f.params[slot4(b, SLOT4_NMU + l)];
            else s = l == 0 ? f.shift4[b].x : l == 1 ? f.shift4[b].y : l == 2 ? f.shift4[b].z : f.shift4[b].w;
            s *= S[0] * inv;   // sum_n r x / N_b: 0 for a component without support
            for (int m = 0; m <= l; ++m) s = __fma_rn(M[4 * l + m], S[1 + m] * inv, s);
            mu[l] = s;
        }
        double v = 0.0;
        if (on)
#pragma unroll
            for (int m = 0; m < 4; ++m) v = __fma_rn(M[4 * i + m], C[4 * m + j], v);
        if (on) A[l] = v;
        __syncwarp();
        // Sigma = A M^T + reg I (symmetric: entry (i, j) computed as (max, min))
        if (on) {
            const int hi = max(i, j), lo = min(i, j);
            v = i == j ? f.reg : 0.0;
#pragma unroll
            for (int m = 0; m < 4; ++m) v = __fma_rn(A[4 * hi + m], M[4 * lo + m], v);
            C[l] = v;
        }
        __syncwarp();
        const double sig = on ? C[l] : 0.0;
        if (on && white && i == j && f.sums == Sums4::Checked) {
            float root = 0.f;
            for (int m = 0; m <= i; ++m) root += fabsf((float)M[4 * i + m]) * sqrtf((float)(S[5 + sym4(m, m)] * inv));
            if (root * rsqrtf((float)sig) > MAX_LOSS4) set_error(st, LOST_SUMS4);
        }
        double fro2 = sig * sig;
#pragma unroll
        for (int o = 8; o > 0; o >>= 1) fro2 += __shfl_xor_sync(FULL, fro2, o);
        // Cholesky by Schur complements, r = the pivots' reciprocal square roots; A = L
        bool pd = true;
        double prod = 1.0;
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            const double piv = on ? C[5 * q] : 1.0;
            pd = pd && piv > 0.0;
            const double u = rsqrt(piv);
            prod *= u;
            if (on && l == 0) r[q] = u;
            if (on && j == q && i >= q) A[l] = C[l] * u;
            __syncwarp();
            if (on && i > q && j > q) C[l] = __fma_rn(-A[4 * i + q], A[4 * j + q], C[l]);
            __syncwarp();
        }
        if (on && !pd && l == 0) {
            atomicMin(&st->bad_component, f.perm ? f.perm[b] : b);
            set_error(st, GIRA_ERR_NOT_PD);
        }
        const bool ok = on && pd;
        // P = L^{-1}
        if (ok) M[l] = i == j ? r[i] : 0.0;
        __syncwarp();
        for (int row = 1; row < 4; ++row) {
            if (ok && i == row && j < row) {
                v = 0.0;
                for (int m = j; m < row; ++m) v = __fma_rn(A[4 * row + m], M[4 * m + j], v);
                M[l] = -v * r[row];
            }
            __syncwarp();
        }
        const float c32 = (float)(log2(nbw * prod) - 2.0 * LOG2_2PI4);
        if (ok) {
            if (j <= i) f.params[slot4(b, SLOT4_P + tri4(i, j))] = (float)(ALPHA4 * M[l]);
            if (l < 4) f.params[slot4(b, SLOT4_NMU + l)] = -(float)mu[l];
            if (l == 4) f.params[slot4(b, SLOT4_C)] = c32;
            if (l == 5) f.params[slot4(b, SLOT4_W)] = (float)nbw;
            if (l == 6) f.params[slot4(b, SLOT4_S)] = sigma_min_sq_bound4(fro2);
            double* m = f.model64 + (size_t)b * MODEL4;
            if (l == 7) m[0] = nbw;
            if (l < 4) m[1 + l] = mu[l];
            if (i <= j) m[5 + sym4(i, j)] = sig;
        }
        if (t == 0 && pp == 0) st->w_raw = 1;
    }
    if (!f.em || pp != 0) return;
    // log-likelihood, trace, convergence (fixed order)
    double v = 0.0;
    if (warp > 0)
        for (int c = t - 32; c < f.ll_count; c += 32 * (FIN4_WARPS - 1)) v += f.llp[c];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(FULL, v, o);
    if (lane == 0) s_ll[warp] = v;
    __syncthreads();
    if (t == 32) {
        v = 0.0;
        for (int w = 1; w < FIN4_WARPS; ++w) v += s_ll[w];
        st->ll_sum = v;
        const double ll = v / (double)f.n;
        f.trace[f.iter - 1] = ll;
        if (f.iter > 1 && fabs(ll - st->prev_ll) < f.tol) st->stop_after = f.iter;
        st->prev_ll = ll;
        st->iters_done = f.iter;
    }
}

// Slot s takes component perm[s]: its row of `old` rebuilt into slot s.
__global__ void rebuild_components4_kernel(const double* __restrict__ old, const int* __restrict__ perm, int k,
                                           double* model64, float* params, DeviceState* st) {
    const int slot = blockIdx.x * blockDim.x + threadIdx.x;
    if (slot >= k) return;
    const int b = perm[slot];
    if (!GIRA_IN(b >= 0 && b < k, st)) return;
    const double* r = old + (size_t)b * MODEL4;
    double S[16];
    for (int i = 0; i < 4; ++i)
        for (int j = 0; j < 4; ++j) S[4 * i + j] = r[5 + sym4(min(i, j), max(i, j))];
    build_component4(slot, r[0], r + 1, S, params, model64, st, b);
}

// Component b of a given model; whether it was built.
__device__ bool build_from_model4(const float* __restrict__ w, const float* __restrict__ mu,
                                  const float* __restrict__ cov, int b, double* model64, float* params,
                                  DeviceState* st) {
    const double pi = w[b];
    double m[4], S[16];
    bool fin = isfinite(pi);
    for (int i = 0; i < 4; ++i) {
        m[i] = mu[4 * (size_t)b + i];
        fin = fin && isfinite(m[i]);
    }
    // the lower triangle is read, as the oracle's Cholesky reads it
    for (int i = 0; i < 4; ++i)
        for (int j = 0; j <= i; ++j) {
            const double v = cov[16 * (size_t)b + 4 * i + j];
            fin = fin && isfinite(v);
            S[4 * i + j] = S[4 * j + i] = v;
        }
    if (!fin) { set_error(st, GIRA_ERR_NONFINITE_INPUT); return false; }
    if (!(pi > 0.0)) { set_error(st, GIRA_ERR_INVALID_ARG); return false; }
    return build_component4(b, pi, m, S, params, model64, st, b);
}

__global__ void params_from_model4_kernel(const float* __restrict__ w, const float* __restrict__ mu,
                                          const float* __restrict__ cov, int k, double* model64, float* params,
                                          float4* ctr, float2* aux, DeviceState* st) {
    const int b = blockIdx.x * blockDim.x + threadIdx.x;
    float c = -INFINITY;
    if (b < k && build_from_model4(w, mu, cov, b, model64, params, st) && ctr) {
        const float* m = mu + 4 * (size_t)b;
        c = params[slot4(b, SLOT4_C)];
        ctr[b] = make_float4(m[0], m[1], m[2], m[3]);
        aux[b] = f2(c, params[slot4(b, SLOT4_S)]);
    }
    if (ctr) raise_cmax(st, c);
}

__global__ void model_out4_kernel(const double* __restrict__ model64, int k, float* w, float* mu, float* cov,
                                  const int* __restrict__ perm, const DeviceState* st) {
    if (st->error) return;         // the given model stays what it was (outputs of a failed call are unspecified)
    __shared__ double s_part[2];   // (the same sum in every block)
    double part = 0.0;
    for (int a2 = threadIdx.x; a2 < k; a2 += blockDim.x) part += model64[(size_t)a2 * MODEL4];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) part += __shfl_xor_sync(FULL, part, o);
    if ((threadIdx.x & 31) == 0) s_part[threadIdx.x >> 5] = part;
    __syncthreads();
    const double nsum = s_part[0] + s_part[1];
    for (int s = blockIdx.x * blockDim.x + threadIdx.x; s < k; s += gridDim.x * blockDim.x) {
        const int b = perm ? perm[s] : s;   // slot s holds the caller's component b
        if (!GIRA_IN(b >= 0 && b < k, const_cast<DeviceState*>(st))) continue;
        const double* m = model64 + (size_t)s * MODEL4;
        w[b] = (float)(st->w_raw ? m[0] / nsum : m[0]);
        for (int i = 0; i < 4; ++i) mu[4 * (size_t)b + i] = (float)m[1 + i];
        for (int i = 0; i < 4; ++i)
            for (int j = 0; j < 4; ++j) cov[16 * (size_t)b + 4 * i + j] = (float)m[5 + sym4(min(i, j), max(i, j))];
    }
}

// Padding components b in [k, kpad): zero parameters, c = -inf.
__global__ void fill_padding4_kernel(float* params, int k, int kpad) {
    const int b = k + blockIdx.x * blockDim.x + threadIdx.x;
    if (b >= kpad) return;
    for (int i = 0; i < PAIR4_FLOATS / 2; ++i) params[slot4(b, i)] = 0.f;
    params[slot4(b, SLOT4_C)] = -INFINITY;
}

// N x 4 -> p4 (x,y,z,I) (nullable) and p8 (x,x,y,y)(z,z,I,I); flags non-finite input.
__global__ void pack4_kernel(const float* __restrict__ p4in, int64_t n, float4* __restrict__ p4,
                             float4* __restrict__ p8, DeviceState* st) {
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const float4 v = make_float4(p4in[4 * i], p4in[4 * i + 1], p4in[4 * i + 2], p4in[4 * i + 3]);
    if (!(isfinite(v.x) && isfinite(v.y) && isfinite(v.z) && isfinite(v.w))) set_error(st, GIRA_ERR_NONFINITE_INPUT);
    if (p4) p4[i] = v;
    p8[2 * i] = make_float4(v.x, v.x, v.y, v.y);
    p8[2 * i + 1] = make_float4(v.z, v.z, v.w, v.w);
}

// ------------------------------------------------------------------ regression of intensity on xyz
// Per component (binary64, then binary32): P_xx = chol(S_xx)^{-1} (6), g = S_xx^{-1} S_xI
// (3), v = S_II - S_Ix g, c = ln pi - sum ln L_ii - (3/2) ln 2 pi, -mu_xyz (3), mu_I, each
// value twice (the operands of packed operations on two locations): slots 0 .. 14; then the
// norms of P_xx's columns (15 .. 17) and a lower bound of sigma_min(P_xx)^2 (18), once each.
constexpr int COND_SLOTS = 20;
constexpr int COND_FLOATS = 2 * COND_SLOTS;   // a component's slots in pairs, read by whole warps
constexpr int COND_ALL = COND_FLOATS + COND_SLOTS;   // + the slots once more, slot i of component b at [i * k + b]:
                                                     // the listing reads 32 components at a time

__global__ void cond_prepare_kernel(const float* __restrict__ w, const float* __restrict__ mu,
                                    const float* __restrict__ cov, int k, float* prep, DeviceState* st) {
    const int b = blockIdx.x * blockDim.x + threadIdx.x;
    if (b >= k) return;
    bool fin = isfinite(w[b]);
    for (int i = 0; i < 4; ++i) fin = fin && isfinite(mu[4 * (size_t)b + i]);
    double S[16];
    for (int i = 0; i < 4; ++i)
        for (int j = 0; j <= i; ++j) {
            S[4 * i + j] = S[4 * j + i] = cov[16 * (size_t)b + 4 * i + j];
            fin = fin && isfinite(S[4 * i + j]);
        }
    if (!fin) {
        set_error(st, GIRA_ERR_NONFINITE_INPUT);
        return;
    }
    double L[9] = {0};
    for (int j = 0; j < 3; ++j) {
        double s = S[4 * j + j];
        for (int kk = 0; kk < j; ++kk) s -= L[3 * j + kk] * L[3 * j + kk];
        if (!(s > 0.0) || !isfinite(s)) {
            atomicMin(&st->bad_component, b);
            set_error(st, GIRA_ERR_NOT_PD);
            return;
        }
        L[3 * j + j] = sqrt(s);
        for (int i = j + 1; i < 3; ++i) {
            double t = S[4 * i + j];
            for (int kk = 0; kk < j; ++kk) t -= L[3 * i + kk] * L[3 * j + kk];
            L[3 * i + j] = t / L[3 * j + j];
        }
    }
    double P[9] = {0};
    for (int c = 0; c < 3; ++c)
        for (int i = c; i < 3; ++i) {
            double t = (i == c) ? 1.0 : 0.0;
            for (int kk = c; kk < i; ++kk) t -= L[3 * i + kk] * P[3 * kk + c];
            P[3 * i + c] = t / L[3 * i + i];
        }
    const double sxi[3] = {S[3], S[7], S[11]};
    double u[3], g[3];
    for (int i = 0; i < 3; ++i) u[i] = P[3 * i] * sxi[0] + P[3 * i + 1] * sxi[1] + P[3 * i + 2] * sxi[2];
    for (int i = 0; i < 3; ++i) g[i] = P[i] * u[0] + P[3 + i] * u[1] + P[6 + i] * u[2];
    const double v = S[15] - (sxi[0] * g[0] + sxi[1] * g[1] + sxi[2] * g[2]);
    const double pi = w[b];
    if (!(pi > 0.0)) { set_error(st, GIRA_ERR_INVALID_ARG); return; }
    const double c = log(pi) - (log(L[0]) + log(L[4]) + log(L[8])) - 1.5 * log(2.0 * 3.14159265358979323846);
    float* o = prep + (size_t)b * COND_FLOATS;
    float* t = prep + (size_t)k * COND_FLOATS + b;
    auto put = [&](int slot, float x) {
        o[2 * slot] = o[2 * slot + 1] = x;
        t[(size_t)slot * k] = x;
    };
    put(0, (float)P[0]); put(1, (float)P[3]); put(2, (float)P[4]); put(3, (float)P[6]); put(4, (float)P[7]);
    put(5, (float)P[8]);
    for (int i = 0; i < 3; ++i) put(6 + i, (float)g[i]);
    put(9, (float)v);
    put(10, (float)c);
    for (int i = 0; i < 3; ++i) put(11 + i, -mu[4 * (size_t)b + i]);
    put(14, mu[4 * (size_t)b + 3]);
    put(15, sqrtf((float)(P[0] * P[0] + P[3] * P[3] + P[6] * P[6])));
    put(16, sqrtf((float)(P[4] * P[4] + P[7] * P[7])));
    put(17, (float)P[8]);
    double fro2 = 0.0;   // lambda_max(S_xx) <= ||S_xx||_F
    for (int i = 0; i < 3; ++i)
        for (int j = 0; j < 3; ++j) fro2 += S[4 * i + j] * S[4 * i + j];
    put(18, 1.f / (sqrtf((float)fro2) * (1.f + 1e-4f)) * (1.f - 1e-4f));
    put(19, 0.f);
}

// Pass 1 takes the maximum log-weight and, as a reference, the regression mean m_ref of that
// component; pass 2 sums w_b = exp(lw_b - max), w_b (m_b - m_ref) and
// w_b (v_b + (m_b - m_ref)^2) in binary32 (the shift keeps the variance free of
// cancellation), both over the components in increasing order.  Two kernels, the same bits.

// Little work: one location per thread, every component, staged through shared memory.  Bound by
// a thread's chain of 2 K components, the same for any order of the locations: up to 38,912
// of them 55 us of kernel for K = 512, where the lists' kernel and the grouping take 85.
constexpr int CD_THREADS = 128;
constexpr int CD_TILE = 64;   // components staged at a time
__global__ void __launch_bounds__(CD_THREADS) conditional4_dense_kernel(const float* __restrict__ locs, int64_t m, int k,
                                                                        const float* __restrict__ prep, float* cmean,
                                                                        float* cvar, DeviceState* st) {
    __shared__ __align__(16) float4 s_rec[CD_TILE][4];   // slots 0 .. 15
    __shared__ int s_err;
    if (threadIdx.x == 0) s_err = st->error;
    __syncthreads();
    if (s_err) return;
    const int64_t i = (int64_t)blockIdx.x * CD_THREADS + threadIdx.x;
    float x[3] = {0.f, 0.f, 0.f};
    if (i < m) {
#pragma unroll
        for (int j = 0; j < 3; ++j) x[j] = locs[3 * i + j];
        if (!(isfinite(x[0]) && isfinite(x[1]) && isfinite(x[2]))) set_error(st, GIRA_ERR_NONFINITE_INPUT);
    }
    // each(o) gets the slots of components 0 .. k - 1
    auto for_all = [&](auto&& each) {
        for (int b0 = 0; b0 < k; b0 += CD_TILE) {
            const int nb = min(CD_TILE, k - b0);
            __syncthreads();
            for (int t = threadIdx.x; t < 16 * nb; t += CD_THREADS)
                reinterpret_cast<float*>(s_rec)[t] = prep[(size_t)(b0 + (t >> 4)) * COND_FLOATS + 2 * (t & 15)];
            __syncthreads();
#pragma unroll 4
            for (int b = 0; b < nb; ++b) {
                float o[16];
#pragma unroll
                for (int q = 0; q < 4; ++q) {
                    const float4 v = s_rec[b][q];
                    o[4 * q] = v.x;
                    o[4 * q + 1] = v.y;
                    o[4 * q + 2] = v.z;
                    o[4 * q + 3] = v.w;
                }
                each(o);
            }
        }
    };
    auto eval = [&](const float (&o)[16], float& mb) {   // log-weight and regression mean
        const float d0 = x[0] + o[11], d1 = x[1] + o[12], d2 = x[2] + o[13];
        const float y0 = o[0] * d0, y1 = fmaf(o[2], d1, o[1] * d0), y2 = fmaf(o[5], d2, fmaf(o[4], d1, o[3] * d0));
        mb = fmaf(o[8], d2, fmaf(o[7], d1, fmaf(o[6], d0, o[14])));
        return fmaf(-0.5f, fmaf(y2, y2, fmaf(y1, y1, y0 * y0)), o[10]);
    };
    float mx = -INFINITY, mref = 0.f;
    for_all([&](const float (&o)[16]) {
        float mb;
        const float lw = eval(o, mb);
        if (lw > mx) {
            mx = lw;
            mref = mb;
        }
    });
    float s = 0.f, e1 = 0.f, e2 = 0.f;
    for_all([&](const float (&o)[16]) {
        float mb;
        const float w = __expf(eval(o, mb) - mx), dm = mb - mref;
        s += w;
        e1 = fmaf(w, dm, e1);
        e2 = fmaf(w, fmaf(dm, dm, o[9]), e2);
    });
    if (i >= m) return;
    if (!(s > 0.f)) {
        set_error(st, GIRA_ERR_NUMERIC);
        return;
    }
    const float inv = 1.f / s, a = e1 * inv;
    cmean[i] = mref + a;
    if (cvar) cvar[i] = fmaf(-a, a, e2 * inv);
}

// More: four warps per 256 locations, neighbours in `order`: a warp has 64 of them, a lane one of
// each block of 32, two locations per packed operation.
// Only components that can matter are visited: exp of less than -104 is exactly 0 in
// binary32, and a term of weight 0 changes no sum.  Over a set of locations, the component
// of largest log-weight at the centre of their box gives every location a log-weight; with L
// the smallest of these, a component whose upper bound over the box (the two bounds of the
// E-step's reach test) is below L - 106 is neither a maximum nor of nonzero weight there.
// Listed first for the 256 locations, by all four warps, then from that list for each warp's
// two blocks (a listing for each warp from all components was two thirds of the time).  The
// listed components' slots go through shared memory, 16 at a time: a block across an edge
// may list hundreds, and their loads one by one are that warp's (and so the kernel's) time.
// Measured: 307,200 locations, K = 1163: 725 us for every component twice, 79 us now (485 us with one
// listing per warp of locations in a depth image's rows).
constexpr int COND_WARPS = 4;
constexpr int COND_CAP = 2048;   // components listed at a time
constexpr int COND_SEG = COND_CAP / COND_WARPS;
constexpr int COND_LOCS = 64;    // locations per warp
constexpr int COND_CHUNK = 16;   // components staged at a time

template <int PER>   // locations per CTA: 256, or one
__global__ void __launch_bounds__(32 * COND_WARPS) conditional4_kernel(const float* __restrict__ locs,
                                                                       const int* __restrict__ order, int64_t m, int k,
                                                                       const float* __restrict__ prep, float* cmean,
                                                                       float* cvar, DeviceState* st) {
    __shared__ __align__(16) float4 s_rec[COND_WARPS][COND_CHUNK][8];
    __shared__ uint16_t s_seg[COND_WARPS][COND_SEG];
    __shared__ uint16_t s_list[COND_WARPS][COND_CAP];
    __shared__ float s_box[COND_WARPS][6], s_bv[COND_WARPS], s_L[COND_WARPS];
    __shared__ int s_bb[COND_WARPS], s_n[COND_WARPS];
    __shared__ int s_err;
    if (threadIdx.x == 0) s_err = st->error;
    __syncthreads();
    if (s_err) return;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    uint16_t* list = s_list[warp];
    const int64_t base = (int64_t)blockIdx.x * PER + warp * COND_LOCS;
    const int64_t end = PER == 1 ? (int64_t)blockIdx.x + 1 : m;
    float x[2][3];   // location base + 32 r + lane
    float lo[2][3], hi[2][3];
#pragma unroll
    for (int r = 0; r < 2; ++r) {
        const int64_t i = min(base + 32 * r + lane, end - 1);   // an absent location: the last one, not written
        const int64_t at = order ? order[i] : i;
        bool fin = true;
#pragma unroll
        for (int j = 0; j < 3; ++j) {
            x[r][j] = locs[3 * at + j];
            fin = fin && isfinite(x[r][j]);
            lo[r][j] = hi[r][j] = x[r][j];
        }
        if (!fin) set_error(st, GIRA_ERR_NONFINITE_INPUT);
#pragma unroll
        for (int o = 16; o > 0; o >>= 1)
#pragma unroll
            for (int j = 0; j < 3; ++j) {
                lo[r][j] = fminf(lo[r][j], __shfl_xor_sync(FULL, lo[r][j], o));
                hi[r][j] = fmaxf(hi[r][j], __shfl_xor_sync(FULL, hi[r][j], o));
            }
    }
    if (lane == 0)
#pragma unroll
        for (int j = 0; j < 3; ++j) {
            s_box[warp][j] = fminf(lo[0][j], lo[1][j]);
            s_box[warp][3 + j] = fmaxf(hi[0][j], hi[1][j]);
        }
    __syncthreads();
    float wlo[3], whi[3];   // the box of all
#pragma unroll
    for (int j = 0; j < 3; ++j) {
        wlo[j] = s_box[0][j];
        whi[j] = s_box[0][3 + j];
#pragma unroll
        for (int w = 1; w < COND_WARPS; ++w) {
            wlo[j] = fminf(wlo[j], s_box[w][j]);
            whi[j] = fmaxf(whi[j], s_box[w][3 + j]);
        }
    }
    const float* soa = prep + (size_t)k * COND_FLOATS;
    auto slot = [&](int b, int i) { return __ldg(soa + (size_t)i * k + b); };
    auto scan_slots = [&](int b, float (&P)[6], float (&nm)[3], float& c) {
#pragma unroll
        for (int i = 0; i < 6; ++i) P[i] = slot(b, i);
#pragma unroll
        for (int i = 0; i < 3; ++i) nm[i] = slot(b, 11 + i);
        c = slot(b, 10);
    };
    auto maha = [&](const float (&P)[6], const float (&d)[3]) {
        const float y0 = P[0] * d[0], y1 = fmaf(P[2], d[1], P[1] * d[0]);
        const float y2 = fmaf(P[5], d[2], fmaf(P[4], d[1], P[3] * d[0]));
        return fmaf(y2, y2, fmaf(y1, y1, y0 * y0));
    };
    auto centre_lw = [&](const float (&P)[6], const float (&nm)[3], float c, const float (&l)[3], const float (&h)[3]) {
        const float d[3] = {0.5f * (l[0] + h[0]) + nm[0], 0.5f * (l[1] + h[1]) + nm[1], 0.5f * (l[2] + h[2]) + nm[2]};
        return fmaf(-0.5f, maha(P, d), c);
    };
    // the upper bound of component b's log-weight over the box
    auto upper = [&](int b, const float (&P)[6], const float (&nm)[3], float c, const float (&l)[3],
                     const float (&u)[3]) {
        const float n0 = slot(b, 15), n1 = slot(b, 16), n2 = slot(b, 17), s2 = slot(b, 18);
        float d[3], h[3], e2 = 0.f;
#pragma unroll
        for (int j = 0; j < 3; ++j) {
            const float ctr = 0.5f * (l[j] + u[j]);
            h[j] = fmaxf(u[j] - ctr, ctr - l[j]);
            d[j] = ctr + nm[j];
            const float e = fmaxf(fabsf(d[j]) - h[j], 0.f);
            e2 = fmaf(e, e, e2);
        }
        const float reach = fmaf(h[0], n0, fmaf(h[1], n1, h[2] * n2));
        const float t = fmaxf(sqrtf(maha(P, d)) * (1.f - 1.f / 256.f) - reach * (1.f + 1.f / 256.f), 0.f);
        const float q = fmaxf(t * t, s2 * e2 * (1.f - 1.f / 128.f));   // <= |P (x - mu)|^2 over the box
        return fmaf(-0.5f, q, c);
    };
    auto warp_best = [&](float& v, int& b) {   // the same choice in every lane
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            const float v2 = __shfl_xor_sync(FULL, v, o);
            const int b2 = __shfl_xor_sync(FULL, b, o);
            if (v2 > v || (v2 == v && b2 < b)) {
                v = v2;
                b = b2;
            }
        }
    };
    auto warp_min = [&](float v) {
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) v = fminf(v, __shfl_xor_sync(FULL, v, o));
        return v;
    };
    auto at_mine = [&](int b, int r) {   // log-weight of component b at this lane's location r
        float P[6], nm[3], c;
        scan_slots(b, P, nm, c);
        const float d[3] = {x[r][0] + nm[0], x[r][1] + nm[1], x[r][2] + nm[2]};
        return fmaf(-0.5f, maha(P, d), c);
    };
    // ---- L of all
    float L_all;
    {
        float v = -INFINITY;
        int best = 0;
        for (int b = threadIdx.x; b < k; b += 32 * COND_WARPS) {
            float P[6], nm[3], c;
            scan_slots(b, P, nm, c);
            const float lw = centre_lw(P, nm, c, wlo, whi);
            if (lw > v) { v = lw; best = b; }
        }
        warp_best(v, best);
        if (lane == 0) {
            s_bv[warp] = v;
            s_bb[warp] = best;
        }
        __syncthreads();
        v = s_bv[0];
        best = s_bb[0];
#pragma unroll
        for (int w = 1; w < COND_WARPS; ++w)
            if (s_bv[w] > v) { v = s_bv[w]; best = s_bb[w]; }
        const float mine = warp_min(fminf(at_mine(best, 0), at_mine(best, 1)));
        if (lane == 0) s_L[warp] = mine;
        __syncthreads();
        L_all = s_L[0];
#pragma unroll
        for (int w = 1; w < COND_WARPS; ++w) L_all = fminf(L_all, s_L[w]);
    }
    // ---- the components of [b0, b1) that this warp's blocks need, in order (called by all warps)
    int nl = 0;
    float known[2] = {-INFINITY, -INFINITY};   // a log-weight of some component at this lane's locations
    auto make_list = [&](int b0, int b1) {
        __syncthreads();   // the segments of the list before this one are read
        const int per = ((b1 - b0 + 32 * COND_WARPS - 1) / (32 * COND_WARPS)) * 32;   // <= COND_SEG
        const int e = min(b1, b0 + per * (warp + 1));
        int n = 0;
        for (int j0 = b0 + per * warp; j0 < e; j0 += 32) {
            const int b = j0 + lane;
            bool want = false;
            if (b < e) {
                float P[6], nm[3], c;
                scan_slots(b, P, nm, c);
                want = !(upper(b, P, nm, c, wlo, whi) < L_all - 106.f);
            }
            const unsigned mk = __ballot_sync(FULL, want);
            if (want) s_seg[warp][n + __popc(mk & ((1u << lane) - 1u))] = (uint16_t)b;
            n += __popc(mk);
        }
        if (lane == 0) s_n[warp] = n;
        __syncthreads();
        int off[COND_WARPS + 1];
        off[0] = 0;
#pragma unroll
        for (int w = 0; w < COND_WARPS; ++w) off[w + 1] = off[w] + s_n[w];
        auto listed = [&](int t) {
            int w = 0, o = 0;
#pragma unroll
            for (int q = 1; q < COND_WARPS; ++q)
                if (t >= off[q]) { w = q; o = off[q]; }
            return (int)s_seg[w][t - o];
        };
        float v[2] = {-INFINITY, -INFINITY}, L[2];
        int best[2] = {-1, -1};
        for (int t = lane; t < off[COND_WARPS]; t += 32) {
            const int b = listed(t);
            float P[6], nm[3], c;
            scan_slots(b, P, nm, c);
#pragma unroll
            for (int r = 0; r < 2; ++r) {
                const float lw = centre_lw(P, nm, c, lo[r], hi[r]);
                if (lw > v[r]) { v[r] = lw; best[r] = b; }
            }
        }
#pragma unroll
        for (int r = 0; r < 2; ++r) {
            warp_best(v[r], best[r]);
            known[r] = best[r] < 0 ? -INFINITY : at_mine(best[r], r);
            L[r] = fmaxf(L_all, warp_min(known[r]));
        }
        nl = 0;
        for (int t0 = 0; t0 < off[COND_WARPS]; t0 += 32) {
            const int t = t0 + lane;
            int b = 0;
            bool want = false;
            if (t < off[COND_WARPS]) {
                b = listed(t);
                float P[6], nm[3], c;
                scan_slots(b, P, nm, c);
#pragma unroll
                for (int r = 0; r < 2; ++r) want = want || !(upper(b, P, nm, c, lo[r], hi[r]) < L[r] - 106.f);
            }
            const unsigned mk = __ballot_sync(FULL, want);
            if (want) list[nl + __popc(mk & ((1u << lane) - 1u))] = (uint16_t)b;
            nl += __popc(mk);
        }
        __syncwarp();
    };
    // the listed components through shared memory; each(o) gets one component's slots in pairs.
    // A list of one chunk that is still there (`staged`) is not loaded again.
    auto for_listed = [&](bool staged, auto&& each) {
        float4 next[COND_CHUNK / 4];   // the chunk after the one in shared memory
        auto fetch = [&](int t0) {
#pragma unroll
            for (int i = 0; i < COND_CHUNK / 4; ++i) {
                const int t = t0 + 4 * i + (lane >> 3);
                if (t < nl)
                    next[i] = __ldg(reinterpret_cast<const float4*>(prep + (size_t)list[t] * COND_FLOATS) + (lane & 7));
            }
        };
        const int total = nl;
        if (!staged) fetch(0);
        for (int t0 = 0; t0 < total; t0 += COND_CHUNK) {
            const int cnt = min(COND_CHUNK, total - t0);
            if (!staged) {
                __syncwarp();
#pragma unroll
                for (int i = 0; i < COND_CHUNK / 4; ++i) s_rec[warp][4 * i + (lane >> 3)][lane & 7] = next[i];
                fetch(t0 + COND_CHUNK);
                __syncwarp();
            }
#pragma unroll 2
            for (int t = 0; t < cnt; ++t) {
                float2 o[16];
#pragma unroll
                for (int i = 0; i < 8; ++i) {
                    const float4 q = s_rec[warp][t][i];
                    o[2 * i] = f2(q.x, q.y);
                    o[2 * i + 1] = f2(q.z, q.w);
                }
                each(o, t0 + t);
            }
        }
    };
    float2 X[3];   // locations of blocks 0, 1
#pragma unroll
    for (int j = 0; j < 3; ++j) X[j] = f2(x[0][j], x[1][j]);
    // log-weights and regression means of component o at two locations (every operation rounds
    // as the scalar one)
    auto eval = [&](const float2 (&o)[16], float2& mb) {
        const float2 d0 = add2(X[0], o[11]), d1 = add2(X[1], o[12]), d2 = add2(X[2], o[13]);
        const float2 y0 = mul2(o[0], d0);
        const float2 y1 = fma2(o[2], d1, mul2(o[1], d0));
        const float2 y2 = fma2(o[5], d2, fma2(o[4], d1, mul2(o[3], d0)));
        mb = fma2(o[8], d2, fma2(o[7], d1, fma2(o[6], d0, o[14])));
        return fma2(dup(-0.5f), fma2(y2, y2, fma2(y1, y1, mul2(y0, y0))), o[10]);
    };
    const bool once = k <= COND_CAP;   // one list serves both passes
    if (once) make_list(0, k);
    const bool cut = once && nl > COND_CHUNK;   // a long list: pass 2 only visits what some location
                                                // needs (one far location makes L low for its block)
    int kept = 0;
    float2 mx = dup(-INFINITY), mref = dup(0.f);
    for (int b0 = 0; b0 < k; b0 += COND_CAP) {
        if (!once) make_list(b0, min(k, b0 + COND_CAP));
        for_listed(false, [&](const float2 (&o)[16], int t) {
            float2 mb;
            const float2 lw = eval(o, mb);
            if (lw.x > mx.x) { mx.x = lw.x; mref.x = mb.x; }
            if (lw.y > mx.y) { mx.y = lw.y; mref.y = mb.y; }
            if (cut) {   // kept <= t: only entries already fetched are overwritten
                const bool want = !(lw.x < fmaxf(mx.x, known[0]) - 106.f) || !(lw.y < fmaxf(mx.y, known[1]) - 106.f);
                if (__any_sync(FULL, want)) {
                    const uint16_t b = list[t];
                    __syncwarp();
                    list[kept++] = b;
                }
            }
        });
    }
    if (cut) nl = kept;
    float2 s = dup(0.f), e1 = dup(0.f), e2 = dup(0.f);
    for (int b0 = 0; b0 < k; b0 += COND_CAP) {
        if (!once) make_list(b0, min(k, b0 + COND_CAP));
        for_listed(once && !cut, [&](const float2 (&o)[16], int) {
            float2 mb;
            const float2 lw = eval(o, mb);
            const float2 w = f2(__expf(lw.x - mx.x), __expf(lw.y - mx.y));
            const float2 dm = f2(mb.x - mref.x, mb.y - mref.y);
            s = add2(s, w);
            e1 = fma2(w, dm, e1);
            e2 = fma2(w, fma2(dm, dm, o[9]), e2);
        });
    }
#pragma unroll
    for (int r = 0; r < 2; ++r) {
        if (base + 32 * r + lane >= end) continue;
        const int64_t i = order ? order[base + 32 * r + lane] : base + 32 * r + lane;
        const float sr = r ? s.y : s.x;
        if (!(sr > 0.f)) {
            set_error(st, GIRA_ERR_NUMERIC);
            continue;
        }
        const float inv = 1.f / sr, a = (r ? e1.y : e1.x) * inv;
        cmean[i] = (r ? mref.y : mref.x) + a;
        if (cvar) cvar[i] = fmaf(-a, a, (r ? e2.y : e2.x) * inv);
    }
}

// ------------------------------------------------------------------ sampling
// Blocks 0 ..: Cholesky factors (binary64, one thread per component).  The last block: the
// cumulative weights in binary64, the running sum in component order.  When every nonzero
// weight is at least 2^-29 and the total below 2, each is a multiple of 2^-52 and every
// partial sum is exact in binary64, whatever the order: a block scan of the integers w 2^52
// gives the same bits as the sequential sum (one thread's chain of K additions, with the
// factors of all components on one SM: 140 us at K = 1163), which the other weights take.
constexpr int SP_THREADS = 256;
__global__ void __launch_bounds__(SP_THREADS) sample_prepare_kernel(const float* __restrict__ w,
                                                                    const float* __restrict__ mu,
                                                                    const float* __restrict__ cov, int k, int d,
                                                                    double* cum, double* chol, DeviceState* st) {
    if (blockIdx.x + 1 < gridDim.x) {
        const int b = blockIdx.x * blockDim.x + threadIdx.x;
        if (b >= k) return;
        bool fin = isfinite(w[b]);
        for (int i = 0; i < d; ++i) fin = fin && isfinite(mu[(size_t)d * b + i]);
        for (int i = 0; i < d * d; ++i) fin = fin && isfinite(cov[(size_t)d * d * b + i]);
        if (!fin) {
            set_error(st, GIRA_ERR_NONFINITE_INPUT);
            return;
        }
        if (!(w[b] >= 0.f)) set_error(st, GIRA_ERR_INVALID_ARG);
        double* L = chol + (size_t)16 * b;
        for (int i = 0; i < 16; ++i) L[i] = 0.0;
        for (int j = 0; j < d; ++j) {
            double s = cov[(size_t)d * d * b + d * j + j];
            for (int kk = 0; kk < j; ++kk) s -= L[4 * j + kk] * L[4 * j + kk];
            if (!(s > 0.0)) {
                atomicMin(&st->bad_component, b);
                set_error(st, GIRA_ERR_NOT_PD);
                break;
            }
            L[4 * j + j] = sqrt(s);
            for (int i = j + 1; i < d; ++i) {
                double t = cov[(size_t)d * d * b + d * i + j];
                for (int kk = 0; kk < j; ++kk) t -= L[4 * i + kk] * L[4 * j + kk];
                L[4 * i + j] = t / L[4 * j + j];
            }
        }
        return;
    }
    __shared__ long long s_sum[SP_THREADS / 32];
    __shared__ int s_bad;
    const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
    const int per = (k + SP_THREADS - 1) / SP_THREADS, b0 = min(k, t * per), b1 = min(k, b0 + per);
    if (t == 0) s_bad = 0;
    __syncthreads();
    long long loc = 0;
    bool ok = true;
    float big = 0.f;
    for (int b = b0; b < b1; ++b) {
        const float x = w[b];
        ok = ok && (x == 0.f || (x >= 0x1p-29f && x < 2.f));
        big += x;
        if (ok) loc += (long long)((double)x * 0x1p52);   // < 2^53 each, at most 8192 of them
    }
    if (!ok || !(big < 2.f)) s_bad = 1;
    long long incl = loc;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const long long v = __shfl_up_sync(FULL, incl, o);
        if (lane >= o) incl += v;
    }
    if (lane == 31) s_sum[warp] = incl;
    __syncthreads();
    long long run = incl - loc, total = 0;
    for (int q = 0; q < SP_THREADS / 32; ++q) {
        if (q < warp) run += s_sum[q];
        total += s_sum[q];
    }
    if (!s_bad && total < (1ll << 53)) {
        for (int b = b0; b < b1; ++b) {
            run += (long long)((double)w[b] * 0x1p52);
            cum[b] = (double)run * 0x1p-52;
        }
        if (t == 0 && total <= 0) set_error(st, GIRA_ERR_INVALID_ARG);
    } else if (t == 0) {
        double tot = 0.0;
        for (int b = 0; b < k; ++b) {
            tot += (double)w[b];
            cum[b] = tot;
        }
        // (a sum that is not finite has a weight that is not: the components' blocks report it)
        if (!(tot > 0.0) && isfinite(tot)) set_error(st, GIRA_ERR_INVALID_ARG);
    }
}

// Sample i: uniforms of draws 5i .. 5i+4 of seed (component, two Box-Muller
// pairs), x = mu_b + L_b z in binary64, rounded to binary32.
__global__ void sample_kernel(int64_t m, int k, int d, const float* __restrict__ mu, const double* __restrict__ cum,
                              const double* __restrict__ chol, uint64_t seed, float* out, int32_t* comp,
                              const DeviceState* st) {
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= m || st->error) return;
    const double tot = cum[k - 1];
    const double u0 = uniform53(seed, 5 * (uint64_t)i) * tot;
    int lo = 0, hi = k - 1;   // first b with cum[b] > u0
    while (lo < hi) {
        const int mid = (lo + hi) >> 1;
        if (cum[mid] > u0) hi = mid; else lo = mid + 1;
    }
    const int b = lo;
    double z[4];
    for (int p = 0; p < 2; ++p) {
        const double u1 = uniform53(seed, 5 * (uint64_t)i + 1 + 2 * p);
        const double u2 = uniform53(seed, 5 * (uint64_t)i + 2 + 2 * p);
        const double r = sqrt(-2.0 * log(1.0 - u1));
        double sn, cs;
        sincos(2.0 * 3.14159265358979323846 * u2, &sn, &cs);
        z[2 * p] = r * cs;
        z[2 * p + 1] = r * sn;
    }
    const double* L = chol + (size_t)16 * b;
    for (int r = 0; r < d; ++r) {
        double x = mu[(size_t)d * b + r];
        for (int c = 0; c <= r; ++c) x += L[4 * r + c] * z[c];
        out[(size_t)d * i + r] = (float)x;
    }
    if (comp) comp[i] = b;
}

// ------------------------------------------------------------------ k-means in four dimensions
// labels = argmin_b ||x - c_b||^2 (binary32 in the order of dist2_f32_4, every operation
// rounded, ties to the lowest b); binary64 sums of the coordinates and counts per label;
// changed[it] counts labels that moved (all of them for it == 0).
// A warp takes 128 consecutive points (Morton order in a fit), four per lane, two centres
// per packed operation.  It scans only the centre pairs that can hold a nearest centre:
// with U an upper bound of every point's nearest distance -- the largest distance to the
// previous centres, or in the first assignment the smallest over the centres of the largest
// distance to the box of the points -- a centre farther than U from the box (with slack for
// the binary32 rounding of both) is farther than that from every point.  The pairs are
// scanned in increasing order, so the argmin and its ties are those of the full scan.  Runs
// of equal labels are summed before the atomics (add_runs).
// Bound by the scan's packed arithmetic and the binary64 sums: 35 us per launch; one point per
// thread over every centre with five binary64 atomics per point took 104 us per launch on
// the 276,348-point frame, K = 512.
constexpr int LL4_THREADS = 256, LL4_PPT = 4;
constexpr int LL4_LIST_MAX = 1024;   // centre pairs up to which the warps keep lists

struct CPair4 {
    float2 c[4];   // negated coordinates of centres 2p and 2p + 1
};

__host__ __device__ constexpr size_t lloyd4_smem(int npair) {
    return sizeof(CPair4) * (size_t)npair + (npair <= LL4_LIST_MAX ? (LL4_THREADS / 32) * (size_t)npair * 2 : 0);
}

template <bool CROWDED>
__global__ void __launch_bounds__(LL4_THREADS) lloyd4_assign_kernel(const float4* __restrict__ pts, int64_t n, int k,
                                                                    const float4* __restrict__ centers,
                                                                    int32_t* labels, double* sums,
                                                                    unsigned long long* changed, int it, float2 nz,
                                                                    DeviceState* st) {
    extern __shared__ CPair4 sc4[];
    if (st->error) return;
    if (it > 0 && changed[it - 1] == 0) return;
    const int npair = (k + 1) / 2;
    for (int p = threadIdx.x; p < npair; p += blockDim.x) {
        const float4 a = centers[2 * p];
        const float4 b = (2 * p + 1 < k) ? centers[2 * p + 1] : make_float4(INFINITY, INFINITY, INFINITY, INFINITY);
        sc4[p].c[0] = f2(-a.x, -b.x);
        sc4[p].c[1] = f2(-a.y, -b.y);
        sc4[p].c[2] = f2(-a.z, -b.z);
        sc4[p].c[3] = f2(-a.w, -b.w);
    }
    __syncthreads();
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    uint16_t* slist = npair <= LL4_LIST_MAX ? reinterpret_cast<uint16_t*>(sc4 + npair) + warp * npair : nullptr;
    unsigned long long cnt = 0;
    constexpr int64_t group = (int64_t)LL4_THREADS * LL4_PPT;
    for (int64_t g0 = (int64_t)blockIdx.x * group; g0 < n; g0 += (int64_t)gridDim.x * group) {
        const int64_t wb = g0 + (int64_t)warp * 32 * LL4_PPT;   // point r of this lane: wb + 4 lane + r
        float2 X[LL4_PPT][4];
        float bd[LL4_PPT];
        int best[LL4_PPT];
#pragma unroll
        for (int r = 0; r < LL4_PPT; ++r) {
            const float4 x = pts[min(wb + LL4_PPT * lane + r, n - 1)];
            X[r][0] = dup(x.x);
            X[r][1] = dup(x.y);
            X[r][2] = dup(x.z);
            X[r][3] = dup(x.w);
            bd[r] = INFINITY;
            best[r] = 0;
        }
        int nl = npair;
        if (slist && wb < n) {
            float lo[4], hi[4];
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                lo[j] = fminf(fminf(X[0][j].x, X[1][j].x), fminf(X[2][j].x, X[3][j].x));
                hi[j] = fmaxf(fmaxf(X[0][j].x, X[1][j].x), fmaxf(X[2][j].x, X[3][j].x));
#pragma unroll
                for (int o = 16; o > 0; o >>= 1) {
                    lo[j] = fminf(lo[j], __shfl_xor_sync(FULL, lo[j], o));
                    hi[j] = fmaxf(hi[j], __shfl_xor_sync(FULL, hi[j], o));
                }
            }
            float U;
            if (it > 0) {
                U = 0.f;
#pragma unroll
                for (int r = 0; r < LL4_PPT; ++r) {
                    const int lp = labels[min(wb + LL4_PPT * lane + r, n - 1)];
                    const CPair4 c = sc4[lp >> 1];
                    float s = 0.f;
#pragma unroll
                    for (int j = 0; j < 4; ++j) {
                        const float d = __fadd_rn(X[r][j].x, (lp & 1) ? c.c[j].y : c.c[j].x);
                        s = __fadd_rn(s, __fmul_rn(d, d));
                    }
                    U = fmaxf(U, s);
                }
#pragma unroll
                for (int o = 16; o > 0; o >>= 1) U = fmaxf(U, __shfl_xor_sync(FULL, U, o));
            } else {
                U = INFINITY;
                for (int b = lane; b < k; b += 32) {
                    const CPair4 c = sc4[b >> 1];
                    float s = 0.f;
#pragma unroll
                    for (int j = 0; j < 4; ++j) {
                        const float nc = (b & 1) ? c.c[j].y : c.c[j].x;
                        const float e = fmaxf(fabsf(lo[j] + nc), fabsf(hi[j] + nc));
                        s = fmaf(e, e, s);
                    }
                    U = fminf(U, s);
                }
#pragma unroll
                for (int o = 16; o > 0; o >>= 1) U = fminf(U, __shfl_xor_sync(FULL, U, o));
            }
            nl = 0;
            for (int j0 = 0; j0 < npair; j0 += 32) {
                const int p = j0 + lane;
                bool live = false;
                if (p < npair) {
                    const CPair4 c = sc4[p];
#pragma unroll
                    for (int m = 0; m < 2; ++m) {   // the centre is -nc
                        float s = 0.f;
#pragma unroll
                        for (int j = 0; j < 4; ++j) {
                            const float nc = m ? c.c[j].y : c.c[j].x;
                            const float e = fmaxf(fmaxf(lo[j] + nc, -nc - hi[j]), 0.f);
                            s = fmaf(e, e, s);
                        }
                        live = live || !(s * (1.f - 1e-5f) > U);
                    }
                }
                const uint32_t mk = __ballot_sync(FULL, live);
                if (live) slist[nl + __popc(mk & ((1u << lane) - 1u))] = (uint16_t)p;
                nl += __popc(mk);
            }
            __syncwarp();
        }
        for (int q = 0; q < nl; ++q) {
            const int p = nl == npair ? q : slist[q];
            const CPair4 c = sc4[p];
#pragma unroll
            for (int r = 0; r < LL4_PPT; ++r) {
                float2 s = f2(0.f, 0.f);
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    const float2 d = add2(X[r][j], c.c[j]);
                    const float2 dd = mul2_alone(d, d, nz);
                    s = j == 0 ? dd : add2(s, dd);
                }
                if (s.x < bd[r]) { bd[r] = s.x; best[r] = 2 * p; }
                if (s.y < bd[r]) { bd[r] = s.y; best[r] = 2 * p + 1; }
            }
        }
        int key[LL4_PPT];
        float x[LL4_PPT][4];
#pragma unroll
        for (int r = 0; r < LL4_PPT; ++r) {
            const int64_t i = wb + LL4_PPT * lane + r;
            key[r] = -1;
            if (i < n) {
                if (it == 0 || labels[i] != best[r]) ++cnt;
                labels[i] = best[r];
                key[r] = best[r];
            }
#pragma unroll
            for (int j = 0; j < 4; ++j) x[r][j] = X[r][j].x;
        }
        add_runs<4, CROWDED>(key, x, sums);
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) cnt += __shfl_xor_sync(FULL, cnt, o);
    if (lane == 0 && cnt) atomicAdd(&changed[it], cnt);
}

__global__ void lloyd4_update_kernel(int k, double* sums, float4* centers, const unsigned long long* changed, int it,
                                     DeviceState* st) {
    if (st->error || changed[it - 1] == 0) return;
    const int b = blockIdx.x * blockDim.x + threadIdx.x;
    if (b < k) {
        double* S = sums + 5 * (size_t)b;
        const double cnt = S[4];
        if (cnt > 0.0)
            centers[b] = make_float4((float)(S[0] / cnt), (float)(S[1] / cnt), (float)(S[2] / cnt), (float)(S[3] / cnt));
        for (int i = 0; i < 5; ++i) S[i] = 0.0;
    }
    if (b == 0) st->lloyd_done = it;
}

// One-hot statistics about the final centres: S0 = count, S1 = sum (x - s),
// S2 = sum (x - s)(x - s)^T, binary64.
// Each thread takes LS4_PPT consecutive points and sums each run of equal labels
// in registers (binary64) before its atomics, as in 3D.
constexpr int LS4_PPT = 8;

__global__ void label_stats4_kernel(const float4* __restrict__ pts, int64_t n, const int32_t* __restrict__ labels,
                                    const float4* __restrict__ shift4, double* stats64, DeviceState* st) {
    if (st->error) return;
    const int64_t step = (int64_t)gridDim.x * blockDim.x * LS4_PPT;
    for (int64_t i0 = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) * LS4_PPT; i0 < n; i0 += step) {
        int key = -1;
        float4 s = make_float4(0.f, 0.f, 0.f, 0.f);
        double a[NSTAT4];
#pragma unroll
        for (int t = 0; t < NSTAT4; ++t) a[t] = 0.0;
        for (int r = 0; r < LS4_PPT; ++r) {
            const int64_t i = i0 + r;
            if (i >= n) break;
            const int b = labels[i];
            if (b != key) {
                if (key >= 0) {
                    double* S = stats64 + (size_t)key * NSTAT4;
#pragma unroll
                    for (int t = 0; t < NSTAT4; ++t) atomicAdd(&S[t], a[t]);
                }
#pragma unroll
                for (int t = 0; t < NSTAT4; ++t) a[t] = 0.0;
                key = b;
                s = shift4[b];
            }
            const float4 x = pts[i];
            const double d[4] = {(double)x.x - (double)s.x, (double)x.y - (double)s.y, (double)x.z - (double)s.z,
                                 (double)x.w - (double)s.w};
            a[0] += 1.0;
#pragma unroll
            for (int t = 0; t < 4; ++t) a[1 + t] += d[t];
#pragma unroll
            for (int i2 = 0; i2 < 4; ++i2)
#pragma unroll
                for (int j = i2; j < 4; ++j) a[5 + sym4(i2, j)] += d[i2] * d[j];
        }
        if (key >= 0) {
            double* S = stats64 + (size_t)key * NSTAT4;
#pragma unroll
            for (int t = 0; t < NSTAT4; ++t) atomicAdd(&S[t], a[t]);
        }
    }
}

}  // namespace

// ------------------------------------------------------------------ launchers
static int num_sms_now() {
    int dev = 0, sms = 1;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    return sms;
}

cudaError_t launch_lloyd4(const float4* pts4, int64_t n, int k, int lloyd_iters, float4* centers, int32_t* labels,
                          double* sums, unsigned long long* changed, DeviceState* st, cudaStream_t s) {
    const float2 nz = make_float2(-0.f, -0.f);
    const size_t smem = lloyd4_smem((k + 1) / 2);
    const int64_t want = (n + (int64_t)LL4_THREADS * LL4_PPT - 1) / ((int64_t)LL4_THREADS * LL4_PPT);
    const int grid = (int)std::max<int64_t>(1, std::min<int64_t>(want, (int64_t)num_sms_now() * 8));
    auto* const assign = k <= CROWDED_LABELS && n > CROWDED_POINTS ? lloyd4_assign_kernel<true> : lloyd4_assign_kernel<false>;
    if (smem > 48 * 1024) {
        const cudaError_t e = cudaFuncSetAttribute(assign, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        if (e != cudaSuccess) return e;
    }
    assign<<<grid, LL4_THREADS, smem, s>>>(pts4, n, k, centers, labels, sums, changed, 0, nz, st);
    for (int it = 1; it <= lloyd_iters; ++it) {
        lloyd4_update_kernel<<<(k + 127) / 128, 128, 0, s>>>(k, sums, centers, changed, it, st);
        assign<<<grid, LL4_THREADS, smem, s>>>(pts4, n, k, centers, labels, sums, changed, it, nz, st);
    }
    return cudaGetLastError();
}

cudaError_t launch_label_stats4(const float4* pts4, int64_t n, int k, const int32_t* labels, const float4* shift4,
                                double* stats64, DeviceState* st, cudaStream_t s) {
    (void)k;
    const int64_t want = (n + 256 * LS4_PPT - 1) / (256 * LS4_PPT);
    const int grid = (int)std::max<int64_t>(1, std::min<int64_t>(want, (int64_t)num_sms_now() * 8));
    label_stats4_kernel<<<grid, 256, 0, s>>>(pts4, n, labels, shift4, stats64, st);
    return cudaGetLastError();
}

// Where the dense E-step is used: up to 10M (point, component)s an iteration of a fit is its two
// launches against five over the lists, and up to 2^24 a log-likelihood's is the shorter chain.
// (More points than 131,072 under few components leave its small CTAs long chains.)  Dense
// and by lists, us: 12 iterations from a given model, 17,000 points, K = 64: 499, 892; 60,000,
// K = 128: 756, 968; 30,000, K = 300: 886, 993; 30,000, K = 550: 1,104, 1,070; 60,000, K = 280:
// 1,176, 1,005; log-likelihood, 17,000, K = 1000: 97, 114; 60,000, K = 280: 95, 101; 250,000,
// K = 64: 95, 101; 276,348, K = 30: 103, 94.  (Models whose components all overlap gain nothing
// from the lists: 100,000 normal points, K = 512, 186 us an iteration dense, 255 by lists.)
bool estep4_dense(int64_t n, int k, bool stats) {
    return k <= MAX_K_DIRECT && n <= 131072 && n * k <= (stats ? 10000000 : 1 << 24);
}

namespace {
int dense4_threads(int k) { return 32 * ((k + 63) / 64); }
}  // namespace

// One wave of CTAs over the points, at most four per SM, and those of one or two warps with 64
// points each (fewer below 8,192 points, where some SMs would be idle): the finalize sums a row
// of every CTA (12 iterations of 17,000 points, K = 64: 475 us with 304 CTAs, 529 with 608,
// 791 with 2,432; 120,000 points: 900, 844, 933).
int estep4_dense_grid(int64_t n, int k, int num_sms, int64_t* ppc) {
    const int threads = dense4_threads(k);
    int occ = 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, estep4_dense_kernel<true>, threads, 0) != cudaSuccess ||
        occ < 1) {
        cudaGetLastError();
        occ = 1;
    }
    const int64_t least = threads <= 64 ? std::min<int64_t>(64, std::max<int64_t>(Q4, n / 128)) : Q4;
    const int64_t grid = std::min<int64_t>((n + least - 1) / least, (int64_t)num_sms * std::min(occ, 4));
    *ppc = std::min<int64_t>(((n + grid - 1) / grid + Q4 - 1) / Q4 * Q4, PPC4_MAX);
    return (int)((n + *ppc - 1) / *ppc);
}

cudaError_t launch_estep4_dense(const EStep4Launch& a, bool stats, int grid, cudaStream_t s, bool pdl) {
    const void* fn = !stats    ? (const void*)estep4_dense_kernel<false>
                     : a.world ? (const void*)estep4_dense_kernel<true, true>
                               : (const void*)estep4_dense_kernel<true>;
    note_estep_kernel(fn);
    void* args[] = {(void*)&a};
    PdlConfig c(dim3(grid), dim3(dense4_threads(a.k)), (size_t)a.pts_per_cta * 32, s, pdl);
    return cudaLaunchKernelExC(&c.cfg, fn, args);
}

cudaError_t launch_reduce_finalize4(const float* partials, const uint32_t* live2, int slices, const double* llp,
                                    int ll_count, const double* stats64, const float4* shift4, int k, int64_t n,
                                    double reg, double tol, double* model64, float* params, double* trace,
                                    const int* perm, DeviceState* st, int iter, bool em, cudaStream_t s, bool pdl,
                                    Sums4 sums) {
    const Fin4Args f{partials, live2, slices, llp, ll_count, stats64, shift4, k, n, reg, tol, model64, params, trace,
                     perm, st, iter, em ? 1 : 0, sums};
    PdlConfig c(dim3((k + 1) / 2), dim3(32 * FIN4_WARPS), 0, s, pdl);
    return cudaLaunchKernelEx(&c.cfg, reduce_finalize4_kernel, f);
}

cudaError_t launch_order_components4(double* model64, double* scratch, int k, int* perm, float* params,
                                     DeviceState* st, cudaStream_t s) {
    cudaError_t e = cudaMemcpyAsync(scratch, model64, sizeof(double) * (size_t)k * MODEL4, cudaMemcpyDeviceToDevice, s);
    if (e == cudaSuccess) e = launch_order_means(scratch, MODEL4, k, perm, s);
    if (e != cudaSuccess) return e;
    rebuild_components4_kernel<<<(k + 63) / 64, 64, 0, s>>>(scratch, perm, k, model64, params, st);
    return cudaGetLastError();
}

cudaError_t launch_params_from_model4(const float* w, const float* mu, const float* cov, int k, double* model64,
                                      float* params, float4* ctr, float2* aux, DeviceState* st, cudaStream_t s) {
    params_from_model4_kernel<<<(k + 63) / 64, 64, 0, s>>>(w, mu, cov, k, model64, params, ctr, aux, st);
    return cudaGetLastError();
}

cudaError_t launch_model_out4(const double* model64, int k, float* w, float* mu, float* cov, const int* perm,
                              const DeviceState* st, cudaStream_t s) {
    model_out4_kernel<<<(k + 63) / 64, 64, 0, s>>>(model64, k, w, mu, cov, perm, st);
    return cudaGetLastError();
}

int params4_pairs(int k) { return (k + 1) / 2; }

cudaError_t launch_fill_padding4(float* params, int k, cudaStream_t s) {
    const int kpad = 2 * params4_pairs(k);
    if (kpad > k) fill_padding4_kernel<<<(kpad - k + 63) / 64, 64, 0, s>>>(params, k, kpad);
    return cudaGetLastError();
}

cudaError_t launch_pack4(const float* pts4in, int64_t n, float4* pts4, float4* pts8, DeviceState* st,
                         cudaStream_t s) {
    pack4_kernel<<<(unsigned)((n + 255) / 256), 256, 0, s>>>(pts4in, n, pts4, pts8, st);
    return cudaGetLastError();
}

int cond_floats() { return COND_ALL; }

// Whether the lists are taken, over 256 neighbouring locations (grouped by cell, 25 us): from 24M
// (location, component)s, with an SM's worth of locations (above 2,048 components, listed in
// rounds, two).  Dense and by lists, us per call (locations of a depth frame): 276,348, K = 8:
// 75, 121; 100,000, K = 100: 91, 120; 30,000, K = 512: 126, 156; 17,000, K = 1163: 190, 211;
// 100,000, K = 300: 139, 142; 60,000, K = 800: 203, 175; 100,000, K = 1163: 353, 220; 30,000,
// K = 3000: 416, 509; 60,000: 580, 511.
bool conditional4_grouped(int64_t m, int k) { return m * k > 24000000 && m > (k <= COND_CAP ? 16384 : 40000); }

cudaError_t launch_conditional4(const float* locs, const int* order, int64_t m, int k, const float* w, const float* mu,
                                const float* cov, float* prep, float* cmean, float* cvar, DeviceState* st,
                                cudaStream_t s) {
    cond_prepare_kernel<<<(k + 63) / 64, 64, 0, s>>>(w, mu, cov, k, prep, st);
    // Few locations under many components: the lists of one location each, a CTA for each, wherever
    // they lie (100 locations all over the frame, K = 1163: 96 us a call, 200 dense, 241 with the
    // lists of 256; 608, K = 128: 83, 87, 88; 2,000, K = 1163: 157, 199, 190).
    if (k >= 64 && m <= std::max(608, std::min(2 * k, 2048))) {
        conditional4_kernel<1><<<(unsigned)m, 32 * COND_WARPS, 0, s>>>(locs, nullptr, m, k, prep, cmean, cvar, st);
        return cudaGetLastError();
    }
    if (!conditional4_grouped(m, k)) {
        conditional4_dense_kernel<<<(unsigned)((m + CD_THREADS - 1) / CD_THREADS), CD_THREADS, 0, s>>>(locs, m, k, prep,
                                                                                                       cmean, cvar, st);
        return cudaGetLastError();
    }
    constexpr int PER = COND_LOCS * COND_WARPS;
    conditional4_kernel<PER><<<(unsigned)((m + PER - 1) / PER), 32 * COND_WARPS, 0, s>>>(locs, order, m, k, prep, cmean,
                                                                                         cvar, st);
    return cudaGetLastError();
}

cudaError_t launch_sample(int64_t m, int k, int d, const float* w, const float* mu, const float* cov, uint64_t seed,
                          double* cum, double* chol, float* out, int32_t* comp, DeviceState* st, cudaStream_t s) {
    sample_prepare_kernel<<<(k + SP_THREADS - 1) / SP_THREADS + 1, SP_THREADS, 0, s>>>(w, mu, cov, k, d, cum, chol, st);
    sample_kernel<<<(unsigned)((m + 127) / 128), 128, 0, s>>>(m, k, d, mu, cum, chol, seed, out, comp, st);
    return cudaGetLastError();
}

}  // namespace gira
