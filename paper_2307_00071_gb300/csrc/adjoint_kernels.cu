// adjoint_kernels.cu -- the gradient of the log-likelihood with every component at every
// point and the statistics about mu_b in world axes: every call on one scan, and batched calls
// that ask for dL/dL_b (Cholesky factors) or have little work (gradient_dense in gira_api.cu has
// the rule and both sides measured).  Other batched calls take the reach lists.
//
// dL/dL_b = lower(P^T (P S2 P^T)) - S0 diag(1/L_ii) multiplies S2 = sum gamma d d^T four
// times by P = L_b^{-1}: for a component thin in one direction (a wall, millimetres against
// decimetres) the binary32 rounding of S2's sums is amplified by the square of its aspect
// ratio, and the value carries up to 1e-4 of it.  Statistics in whitened coordinates, as the
// reach lists keep them, are an order of magnitude closer to 64-bit results there, but no
// finish of dL/dL_b from them exists, and its values would move by that rounding.  A call on one
// scan gives the same bits whichever gradients it asks for.
//
// Mapping (component-stationary): one CTA holds all K <= 1024 components, spread over its
// warps; lane l of warp w owns NP component pairs in registers.  All lanes walk the CTA's
// contiguous range of points together, Q at a time: pass 1 computes e for the lane's
// components, the per-point sums are combined across lanes (shuffle transpose-reduce) and
// warps (shared memory), and pass 2 accumulates S0 = sum r, S1 = sum r d, S2 = sum r d d^T
// (binary32, per-CTA partials) and each point's sum over components of gamma Sigma_b^{-1} d.
#include <float.h>
#include <math.h>

#include <algorithm>

#include "gira_internal.cuh"

namespace gira {

namespace {

constexpr unsigned FULL = 0xffffffffu;
constexpr double LN2 = 0.693147180559945309417232121458;
constexpr int FIN_CPB = 2;          // components per block of the sums
constexpr int FIN_SPLIT_CTA = 16;   // per-CTA partials: one output summed in 16 fixed slices
constexpr int FIN_THREADS = FIN_CPB * NSTAT * FIN_SPLIT_CTA;   // 320

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


constexpr long long MBAR_POLL_LIMIT = 2000000000ll;   // bound on any mbarrier wait: 2 s of wall time
constexpr int PPC_MAX = 2048;                         // points staged per CTA (64 KB)
constexpr int QB = 8;                                 // points per batch

// The CTA's points arrive in one TMA bulk copy, laid out (x,x,y,y)(z,z,0,0) per point.  Per
// batch of Q points: pass 1 (logits, e, warp-level sums), one CTA barrier, the cross-warp
// total and 1/total, pass 2, a second barrier, the point gradients dL/dx' = -(2 ln 2) sum
// gamma P'^T P' d.  The per-point sums are double-buffered by batch parity: a warp can only
// overwrite a buffer after the next barrier, which every warp reaches after reading it.  The
// owner lanes write dL/dx = R^T dL/dx' and accumulate the pose sums (dL/dx' x'^T, dL/dx').
// Measured: 100k points, K = 1024: 266 to 274 us for a scan on its model, 313 to 339 us for one 0.1 to
// 0.5 m off it (points more than 100 binades below the reference take the exact maximum).
template <int NP, int Q, int MAXT, int MINB, bool GRAD>
__global__ void __launch_bounds__(MAXT, MINB) estep_adjoint_kernel(const AdjointLaunch a_in) {
    extern __shared__ __align__(128) unsigned char dsm[];
    __shared__ __align__(8) uint64_t bar_tma;
    __shared__ float red_sum[2][32][Q];
    __shared__ float red_g[GRAD ? 2 : 1][GRAD ? 32 : 1][Q][3];
    __shared__ float red_aux[2][32][Q];
    __shared__ float s_cmax[32], s_wsum[32];
    __shared__ int s_skip, s_norm, s_dead;
    constexpr int LPQ = 32 / Q;   // lanes per batch index after the transpose-reduce

    // batched launches: this CTA's instance and CTA index within it
    int cta = blockIdx.x;
    AdjointLaunch a = a_in;
    if (a_in.units) {
        const BatchUnit u = a_in.units[blockIdx.x];
        const BatchInst I = a_in.insts[u.inst];
        cta = u.cta;
        a.pts8 = a_in.pts8 + 2 * I.pt_off;
        a.n = I.n;
        a.k = I.k;
        a.params = a_in.params + I.par_off;
        a.pts_per_cta = I.ppc;
        a.partials = a_in.partials ? a_in.partials + I.part_off : nullptr;
        a.ll_partials = a_in.ll_partials + I.ll_off;
        a.st = a_in.states + u.inst;
        // per-instance scan gradient rows, pose and pose sums
        a.grad_pts = a_in.grad_pts ? a_in.grad_pts + 3 * I.pt_off : nullptr;
        a.rot = a_in.rot ? a_in.rot + 12 * (size_t)u.inst : nullptr;
        a.pose_partials = a_in.pose_partials + 12 * I.ll_off;
    }
    const int G = blockDim.x >> 5;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int64_t begin = (int64_t)cta * a.pts_per_cta;
    const int64_t end = min(a.n, begin + a.pts_per_cta);
    const int npts = (int)(end - begin);
    const int nb = (npts + Q - 1) / Q;
    const float4* spts = reinterpret_cast<const float4*>(dsm);
    if (threadIdx.x == 0) {
        // the points are never written by the kernel this one may overlap
        // (dependent launch), so their copy starts before the wait below
        mbar_init(&bar_tma, 1);
        mbar_fence_init();
        mbar_expect_tx(&bar_tma, (uint32_t)npts * 32u);
        tma_load_1d(reinterpret_cast<void*>(dsm), a.pts8 + 2 * begin, (uint32_t)npts * 32u, &bar_tma);
    }
    pdl_wait();   // the parameters and the state written by the previous kernel
    if (threadIdx.x == 0) {
        s_skip = (a.iter > a.st->stop_after) || (a.st->error != 0);
        s_norm = a.st->w_raw;
        s_dead = 0;
    }
    __syncthreads();
    if (s_skip) {   // let the copy land before leaving
        if (threadIdx.x == 0) mbar_wait_bounded(&bar_tma, 0u, MBAR_POLL_LIMIT);
        return;
    }
    pdl_allow_next();

    // ---- this lane's component pairs -> registers (overlaps the TMA)
    PairParams prm[NP];
    float cm = -INFINITY, ws = 0.f;
#pragma unroll
    for (int j = 0; j < NP; ++j) {
        const int pp = (warp * NP + j) * 32 + lane;
        const float4* src = reinterpret_cast<const float4*>(a.params + (size_t)pp * PAIR_FLOATS);
        const float4 v0 = src[0], v1 = src[1], v2 = src[2], v4 = src[4], v5 = src[5], v6 = src[6];
        prm[j].p[0] = f2(v0.x, v0.y); prm[j].p[1] = f2(v0.z, v0.w);
        prm[j].p[2] = f2(v1.x, v1.y); prm[j].p[3] = f2(v1.z, v1.w);
        prm[j].p[4] = f2(v2.x, v2.y); prm[j].p[5] = f2(v2.z, v2.w);
        prm[j].c = f2(v4.z, v4.w);
        prm[j].nmu[0] = f2(v5.x, v5.y); prm[j].nmu[1] = f2(v5.z, v5.w);
        prm[j].nmu[2] = f2(v6.x, v6.y);
        cm = fmaxf(cm, fmaxf(prm[j].c.x, prm[j].c.y));
        ws += v6.z + v6.w;
    }
    // reference cmax = max_b c_b >= every logit (every e <= 1); after an M-step
    // also the weight normaliser sum_a N_a (shifts the log-likelihood only)
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        cm = fmaxf(cm, __shfl_xor_sync(FULL, cm, o));
        ws += __shfl_xor_sync(FULL, ws, o);
    }
    if (lane == 0) {
        s_cmax[warp] = cm;
        s_wsum[warp] = ws;
    }
    if (!mbar_wait_bounded(&bar_tma, 0u, MBAR_POLL_LIMIT)) s_dead = 1;
    __syncthreads();
    if (s_dead) {   // the points never arrived: report, let the copy land, leave
        if (threadIdx.x == 0) {
            set_error(a.st, GIRA_ERR_TIMEOUT);
            mbar_wait_bounded(&bar_tma, 0u, MBAR_POLL_LIMIT);
        }
        return;
    }
    float cmax = s_cmax[0], wsum = s_wsum[0];
    for (int w = 1; w < G; ++w) {
        cmax = fmaxf(cmax, s_cmax[w]);
        wsum += s_wsum[w];
    }
    const float ref0 = s_norm ? cmax - __log2f(wsum) : cmax;
#pragma unroll
    for (int j = 0; j < NP; ++j) prm[j].c = f2(cmax - prm[j].c.x, cmax - prm[j].c.y);

    float Sx[NP][NSTAT], Sy[NP][NSTAT];   // statistics of components 2p and 2p+1
    if (GRAD)
#pragma unroll
        for (int j = 0; j < NP; ++j)
#pragma unroll
            for (int s = 0; s < NSTAT; ++s) Sx[j][s] = Sy[j][s] = 0.f;
    double ll_acc = 0.0;
    const int myq = q_of_lane<Q>(lane);
    const bool owner = (warp == 0) && ((lane & (LPQ - 1)) == 0);

    auto load_pt = [&](int li, float2& X0, float2& X1, float2& X2) {
        const float4 xy = spts[2 * li], zz = spts[2 * li + 1];
        X0 = f2(xy.x, xy.y);
        X1 = f2(xy.z, xy.w);
        X2 = f2(zz.x, zz.y);
    };
    // pass 1 of batch t: e for every (point, own component) into E, warp-level sums into red_sum[t & 1]
    auto pass1 = [&](int t, float2 (&E)[NP][Q]) {
        const int lb = t * Q, nvalid = min(Q, npts - lb);
        float part[Q];
#pragma unroll
        for (int q = 0; q < Q; ++q) {
            float2 X0, X1, X2;
            load_pt((q < nvalid) ? lb + q : lb, X0, X1, X2);
            float2 acc = f2(0.f, 0.f);
#pragma unroll
            for (int j = 0; j < NP; ++j) {
                const float2 nq = neg_logit2(prm[j], X0, X1, X2);
                const float2 e = f2(ex2_approx(0.f - nq.x), ex2_approx(0.f - nq.y));
                E[j][q] = e;
                acc = add2(acc, e);
            }
            part[q] = acc.x + acc.y;
        }
        const float wt = warp_transpose_reduce<Q>(part, lane, AddOp());
        if ((lane & (LPQ - 1)) == 0) red_sum[t & 1][warp][myq] = wt;
    };
    // statistics of batch t from E and the reciprocal sums r (owned by lane q * LPQ)
    auto pass2 = [&](int t, const float2 (&E)[NP][Q], float r) {
        const int lb = t * Q, nvalid = min(Q, npts - lb);
        float gq[Q][3];   // this lane's share of sum_b gamma P'^T P' d, per point
#pragma unroll
        for (int q = 0; q < Q; ++q) {
            gq[q][0] = gq[q][1] = gq[q][2] = 0.f;
            // pairs with a nonzero e for this point on some lane of the warp (warp-uniform)
            bool live[NP], any = false;
#pragma unroll
            for (int j = 0; j < NP; ++j) {
                live[j] = __any_sync(FULL, (E[j][q].x != 0.f) || (E[j][q].y != 0.f));
                any = any || live[j];
            }
            if (!any) continue;
            float2 X0, X1, X2;
            load_pt((q < nvalid) ? lb + q : lb, X0, X1, X2);
            const float R = __shfl_sync(FULL, r, q * LPQ);
            // scalar FP32: measured faster than the packed form for this
            // accumulate-heavy pattern
            auto acc1 = [&](float e, float m0, float m1, float m2, float (&T)[NSTAT], const float2 (&pp)[6], int h) {
                const float g = e * R;
                const float d0 = X0.x + m0, d1 = X1.x + m1, d2 = X2.x + m2;
                {
                    const float p0 = h ? pp[0].y : pp[0].x, p1 = h ? pp[1].y : pp[1].x, p2 = h ? pp[2].y : pp[2].x;
                    const float p3 = h ? pp[3].y : pp[3].x, p4 = h ? pp[4].y : pp[4].x, p5 = h ? pp[5].y : pp[5].x;
                    const float y0 = p0 * d0, y1 = fmaf(p2, d1, p1 * d0), y2 = fmaf(p5, d2, fmaf(p4, d1, p3 * d0));
                    const float z0 = fmaf(p3, y2, fmaf(p1, y1, p0 * y0)), z1 = fmaf(p4, y2, p2 * y1), z2 = p5 * y2;
                    gq[q][0] = fmaf(g, z0, gq[q][0]);
                    gq[q][1] = fmaf(g, z1, gq[q][1]);
                    gq[q][2] = fmaf(g, z2, gq[q][2]);
                }
                const float g0 = g * d0, g1 = g * d1, g2 = g * d2;
                T[0] += g;
                T[1] += g0;
                T[2] += g1;
                T[3] += g2;
                T[4] = fmaf(g0, d0, T[4]);
                T[5] = fmaf(g0, d1, T[5]);
                T[6] = fmaf(g0, d2, T[6]);
                T[7] = fmaf(g1, d1, T[7]);
                T[8] = fmaf(g1, d2, T[8]);
                T[9] = fmaf(g2, d2, T[9]);
            };
#pragma unroll
            for (int j = 0; j < NP; ++j) {
                if (!live[j]) continue;
                acc1(E[j][q].x, prm[j].nmu[0].x, prm[j].nmu[1].x, prm[j].nmu[2].x, Sx[j], prm[j].p, 0);
                acc1(E[j][q].y, prm[j].nmu[0].y, prm[j].nmu[1].y, prm[j].nmu[2].y, Sy[j], prm[j].p, 1);
            }
        }
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            float v[Q];
#pragma unroll
            for (int q = 0; q < Q; ++q) v[q] = gq[q][c];
            const float w = warp_transpose_reduce<Q>(v, lane, AddOp());
            if ((lane & (LPQ - 1)) == 0) red_g[t & 1][warp][myq][c] = w;
        }
    };
    // batch t after its barrier: cross-warp total, rare exact-max path, 1/total
    auto finish = [&](int t, float2 (&E)[NP][Q]) -> float {
        const int lb = t * Q, nvalid = min(Q, npts - lb);
        float tot = red_sum[t & 1][0][myq];
        for (int w = 1; w < G; ++w) tot += red_sum[t & 1][w][myq];
        const bool myvalid = myq < nvalid;
        float ref = ref0;
        // Rare path: a point whose best component is > 100 binades below cmax.
        // Redo the batch with the exact per-point maximum (Eq. logestep's
        // max-subtraction) so that no responsibility is lost to underflow.
        if (__any_sync(FULL, myvalid && !(tot >= 0x1p-100f))) {
            float m[Q];
#pragma unroll
            for (int q = 0; q < Q; ++q) {
                float2 X0, X1, X2;
                load_pt((q < nvalid) ? lb + q : lb, X0, X1, X2);
                float mm = -INFINITY;
#pragma unroll
                for (int j = 0; j < NP; ++j) {
                    const float2 nq = neg_logit2(prm[j], X0, X1, X2);
                    const float2 l = f2(-nq.x, -nq.y);
                    E[j][q] = l;
                    mm = fmaxf(mm, fmaxf(l.x, l.y));
                }
                m[q] = mm;
            }
            float mt = warp_transpose_reduce<Q>(m, lane, MaxOp());
            if ((lane & (LPQ - 1)) == 0) red_aux[0][warp][myq] = mt;
            __syncthreads();
            mt = red_aux[0][0][myq];
            for (int w = 1; w < G; ++w) mt = fmaxf(mt, red_aux[0][w][myq]);
            float part[Q];
#pragma unroll
            for (int q = 0; q < Q; ++q) {
                float mq = __shfl_sync(FULL, mt, q * LPQ);
                mq = (mq > -INFINITY) ? mq : 0.f;
                float2 acc = f2(0.f, 0.f);
#pragma unroll
                for (int j = 0; j < NP; ++j) {
                    const float2 e = f2(ex2_approx(E[j][q].x - mq), ex2_approx(E[j][q].y - mq));
                    E[j][q] = e;
                    acc = add2(acc, e);
                }
                part[q] = acc.x + acc.y;
            }
            const float wt = warp_transpose_reduce<Q>(part, lane, AddOp());
            if ((lane & (LPQ - 1)) == 0) red_aux[1][warp][myq] = wt;
            __syncthreads();
            tot = red_aux[1][0][myq];
            for (int w = 1; w < G; ++w) tot += red_aux[1][w][myq];
            if (myvalid && !(mt > -INFINITY)) set_error(a.st, GIRA_ERR_NUMERIC);
            ref = ref0 + ((mt > -INFINITY) ? mt : 0.f);
        }
        const bool ok = myvalid && tot > 0.f;
        const float lse2 = lg2_approx(tot) + ref;   // log2 sum_b pi_b N(x|b)
        if (owner && ok) ll_acc += (double)lse2;
        return ok ? __frcp_rn(tot) : 0.f;
    };
    float2 E[NP][Q];
    float tw[12] = {};   // owner lanes: sum g x'^T (row-major), sum g
    for (int t = 0; t < nb; ++t) {
        pass1(t, E);
        __syncthreads();   // every warp's sums of batch t are in red_sum[t & 1]
        const float r = finish(t, E);
        if (GRAD) {
            pass2(t, E, r);
            __syncthreads();   // every warp's gradient sums of batch t are in red_g[t & 1]
            const int lb = t * Q;
            if (owner && myq < min(Q, npts - lb)) {
                float g3[3];
#pragma unroll
                for (int c = 0; c < 3; ++c) {
                    float v = red_g[t & 1][0][myq][c];
                    for (int w = 1; w < G; ++w) v += red_g[t & 1][w][myq][c];
                    g3[c] = -1.38629436111989061883f * v;   // -(2 ln 2): P'^T P' = Sigma^{-1} log2(e) / 2
                }
                const float4 xy = spts[2 * (lb + myq)], zz = spts[2 * (lb + myq) + 1];
                const float x0 = xy.x, x1 = xy.z, x2 = zz.x;
                const float xq[3] = {x0, x1, x2};
#pragma unroll
                for (int i = 0; i < 3; ++i) {
#pragma unroll
                    for (int j = 0; j < 3; ++j) tw[3 * i + j] = fmaf(g3[i], xq[j], tw[3 * i + j]);
                    tw[9 + i] += g3[i];
                }
                if (a.grad_pts) {
                    float* gp = a.grad_pts + 3 * (begin + lb + myq);
                    if (a.rot) {
                        const float* Rm = a.rot;
                        gp[0] = fmaf(Rm[6], g3[2], fmaf(Rm[3], g3[1], Rm[0] * g3[0]));
                        gp[1] = fmaf(Rm[7], g3[2], fmaf(Rm[4], g3[1], Rm[1] * g3[0]));
                        gp[2] = fmaf(Rm[8], g3[2], fmaf(Rm[5], g3[1], Rm[2] * g3[0]));
                    } else {
                        gp[0] = g3[0];
                        gp[1] = g3[1];
                        gp[2] = g3[2];
                    }
                }
            }
        }
    }

    if (GRAD) {
        float* dst = a.partials + (size_t)cta * a.k * NSTAT;
#pragma unroll
        for (int j = 0; j < NP; ++j) {
            const int b0 = 2 * ((warp * NP + j) * 32 + lane);
            if (b0 < a.k)
#pragma unroll
                for (int s = 0; s < NSTAT; ++s) dst[(size_t)b0 * NSTAT + s] = Sx[j][s];
            if (b0 + 1 < a.k)
#pragma unroll
                for (int s = 0; s < NSTAT; ++s) dst[(size_t)(b0 + 1) * NSTAT + s] = Sy[j][s];
        }
    }
    if (warp == 0) {   // owner lanes hold the per-point log-likelihood sums; fixed order
        double v = ll_acc;
#pragma unroll
        for (int o = LPQ; o < 32; o <<= 1) v += __shfl_xor_sync(FULL, v, o);
        if (lane == 0) a.ll_partials[cta] = v * LN2;
        if (GRAD) {
#pragma unroll
            for (int i = 0; i < 12; ++i) {
                double u = owner ? (double)tw[i] : 0.0;
#pragma unroll
                for (int o = LPQ; o < 32; o <<= 1) u += __shfl_xor_sync(FULL, u, o);
                if (lane == 0) a.pose_partials[(size_t)cta * 12 + i] = u;
            }
        }
    }
}

// The statistics of components b0 .. b0 + nout / NSTAT - 1 summed over the
// per-CTA partials into S (binary64): FIN_SPLIT_CTA fixed slices of CTAs, binary32
// groups of 8 within a slice, binary64 across groups and slices.  Call with
// every thread of the block; ends with S valid after a barrier.
__device__ void reduce_partials(const float* __restrict__ partials, int grid, int k, int b0, int nout,
                                double (*part)[FIN_CPB * NSTAT], double* S) {
    const int t = threadIdx.x;
    const int o = t % (FIN_CPB * NSTAT), q = t / (FIN_CPB * NSTAT);
    if (o < nout) {
        const int c0 = q * grid / FIN_SPLIT_CTA, c1 = (q + 1) * grid / FIN_SPLIT_CTA;
        const float* src = partials + (size_t)b0 * NSTAT + o;
        const size_t stride = (size_t)k * NSTAT;
        double acc = 0.0;
        for (int c = c0; c < c1; c += 8) {   // eight independent loads in flight
            float v[8];
#pragma unroll
            for (int u = 0; u < 8; ++u) v[u] = (c + u < c1) ? __ldcg(src + (size_t)(c + u) * stride) : 0.f;
            float f = 0.f;
#pragma unroll
            for (int u = 0; u < 8; ++u) f += v[u];
            acc += (double)f;
        }
        part[q][o] = acc;
    }
    __syncthreads();
    if (t < nout) {
        double v = 0.0;
        for (int q2 = 0; q2 < FIN_SPLIT_CTA; ++q2) v += part[q2][t];
        S[t] = v;
    }
}

// Parameter gradients from the statistics about mu_b (d = x' - mu_b):
//   dL/dmu_b    = Sigma^{-1} S1 = P^T P S1
//   dL/dL_b     = lower(P^T (P S2 P^T) - S0 diag(1/L_ii))
//   dL/dalpha_b = S0 - N pi_b
// with P = L_b^{-1}; block 0 also sums the log-likelihood and the twist.
__device__ void grad_finalize_body(const AdjointFinArgs& f, int blk);
__global__ void __launch_bounds__(FIN_THREADS) grad_finalize_kernel(const AdjointFinArgs f) {
    grad_finalize_body(f, blockIdx.x);
}
// Block (instance i, index j) of a batch: components j * FIN_CPB .. of instance i.
__global__ void __launch_bounds__(FIN_THREADS) grad_finalize_batched_kernel(const AdjointFinArgs base,
                                                                           const BatchInst* __restrict__ insts,
                                                                           const int2* __restrict__ blocks,
                                                                           DeviceState* states) {
    const int2 bi = blocks[blockIdx.x];
    const BatchInst I = insts[bi.x];
    const size_t c = I.comp_off;
    AdjointFinArgs f = base;
    f.partials = base.partials + I.part_off;
    f.grid = I.ctas;
    f.llp = base.llp + I.ll_off;
    f.pp = base.pp + 12 * I.ll_off;
    f.pose = base.pose ? base.pose + 12 * (size_t)bi.x : nullptr;
    f.chol = base.chol + 9 * c;
    f.model64 = base.model64 + c * MODEL;
    f.k = I.k;
    f.n = I.n;
    f.g_logits = base.g_logits ? base.g_logits + c : nullptr;
    f.g_means = base.g_means ? base.g_means + 3 * c : nullptr;
    f.g_chol = base.g_chol ? base.g_chol + 9 * c : nullptr;
    f.g_pose = base.g_pose ? base.g_pose + 12 * (size_t)bi.x : nullptr;
    f.g_twist = base.g_twist ? base.g_twist + 6 * (size_t)bi.x : nullptr;
    f.st = states + bi.x;
    grad_finalize_body(f, bi.y);
}
__device__ void grad_finalize_body(const AdjointFinArgs& f, int blk) {
    __shared__ double part[FIN_SPLIT_CTA][FIN_CPB * NSTAT];
    __shared__ double S[FIN_CPB * NSTAT];
    __shared__ int s_skip;
    const float* __restrict__ partials = f.partials;
    const int grid = f.grid;
    const double* __restrict__ llp = f.llp;
    const double* __restrict__ pp = f.pp;
    const float* __restrict__ pose = f.pose;
    const float* __restrict__ chol = f.chol;
    const double* __restrict__ model64 = f.model64;
    const int k = f.k;
    const int64_t n = f.n;
    float* g_logits = f.g_logits;
    float* g_means = f.g_means;
    float* g_chol = f.g_chol;
    double* g_pose = f.g_pose;
    double* g_twist = f.g_twist;
    DeviceState* st = f.st;
    if (threadIdx.x == 0) s_skip = st->error != 0;
    __syncthreads();
    if (s_skip) return;
    const int t = threadIdx.x;
    const int b0 = blk * FIN_CPB;
    const int nb = min(FIN_CPB, k - b0);
    reduce_partials(partials, grid, k, b0, nb * NSTAT, part, S);
    __syncthreads();
    if (t < nb) {
        const int b = b0 + t;
        const double* Sb = S + t * NSTAT;
        const float* L = chol + 9 * (size_t)b;
        const double L00 = L[0], L10 = L[3], L11 = L[4], L20 = L[6], L21 = L[7], L22 = L[8];
        const double P00 = 1.0 / L00, P11 = 1.0 / L11, P22 = 1.0 / L22;
        const double P10 = -L10 * P00 * P11, P21 = -L21 * P11 * P22, P20 = -(L20 * P00 + L21 * P10) * P22;
        const double P[3][3] = {{P00, 0.0, 0.0}, {P10, P11, 0.0}, {P20, P21, P22}};
        const double s0 = Sb[0];
        const double s1[3] = {Sb[1], Sb[2], Sb[3]};
        const double S2[3][3] = {{Sb[4], Sb[5], Sb[6]}, {Sb[5], Sb[7], Sb[8]}, {Sb[6], Sb[8], Sb[9]}};
        double u[3], gm[3];
        for (int i = 0; i < 3; ++i) u[i] = P[i][0] * s1[0] + P[i][1] * s1[1] + P[i][2] * s1[2];
        for (int i = 0; i < 3; ++i) gm[i] = P[0][i] * u[0] + P[1][i] * u[1] + P[2][i] * u[2];
        double A[3][3], M[3][3];   // A = P S2, M = A P^T
        for (int i = 0; i < 3; ++i)
            for (int j = 0; j < 3; ++j) A[i][j] = P[i][0] * S2[0][j] + P[i][1] * S2[1][j] + P[i][2] * S2[2][j];
        for (int i = 0; i < 3; ++i)
            for (int j = 0; j < 3; ++j) M[i][j] = A[i][0] * P[j][0] + A[i][1] * P[j][1] + A[i][2] * P[j][2];
        const double Ld[3] = {L00, L11, L22};
        for (int i = 0; i < 3; ++i) {
            for (int j = 0; j < 3; ++j) {
                double v = 0.0;
                if (j <= i) {
                    v = P[0][i] * M[0][j] + P[1][i] * M[1][j] + P[2][i] * M[2][j];
                    if (i == j) v -= s0 / Ld[i];
                }
                if (g_chol) g_chol[9 * (size_t)b + 3 * i + j] = (float)v;
            }
            if (g_means) g_means[3 * (size_t)b + i] = (float)gm[i];
        }
        if (g_logits) g_logits[b] = (float)(s0 - (double)n * model64[(size_t)b * MODEL]);
    }
    if (blk == 0 && t >= 32 && t < 64) {   // warp 1: log-likelihood and pose sums, fixed order
        const int lane = t - 32;
        double v[13] = {};
        for (int c = lane; c < grid; c += 32) {
            v[0] += llp[c];
            for (int i = 0; i < 12; ++i) v[1 + i] += pp[(size_t)c * 12 + i];
        }
        for (int i = 0; i < 13; ++i) {
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) v[i] += __shfl_xor_sync(FULL, v[i], o);
        }
        if (lane == 0) {
            st->ll_sum = v[0];
            const double* M = v + 1;    // sum g x'^T
            const double* G = v + 10;   // sum g
            if (g_twist) {   // omega = sum x' x g, v = sum g
                g_twist[0] = M[3 * 2 + 1] - M[3 * 1 + 2];
                g_twist[1] = M[3 * 0 + 2] - M[3 * 2 + 0];
                g_twist[2] = M[3 * 1 + 0] - M[3 * 0 + 1];
                for (int i = 0; i < 3; ++i) g_twist[3 + i] = G[i];
            }
            if (g_pose) {    // x = R^T (x' - t): dL/dR = (sum g x'^T - G t^T) R, dL/dt = G
                const double tt[3] = {pose ? pose[9] : 0.0, pose ? pose[10] : 0.0, pose ? pose[11] : 0.0};
                for (int i = 0; i < 3; ++i)
                    for (int j = 0; j < 3; ++j) {
                        double acc = 0.0;
                        for (int m = 0; m < 3; ++m) {
                            const double Rmj = pose ? (double)pose[3 * m + j] : (m == j ? 1.0 : 0.0);
                            acc += (M[3 * i + m] - G[i] * tt[m]) * Rmj;
                        }
                        g_pose[3 * i + j] = acc;
                    }
                for (int i = 0; i < 3; ++i) g_pose[9 + i] = G[i];
            }
        }
    }
}

// Shapes: K <= 64 -> one component pair per lane and one warp; otherwise two pairs per lane
// and ceil(K / 128) warps.
struct Shape {
    int np, g, threads;
};
Shape shape_for(int k) {
    if (k <= 64) return {1, 1, 32};
    const int g = (k + 127) / 128;
    return {2, g, 32 * g};
}
const void* kernel_for(const Shape& sh, bool grad) {
    if (!grad) {
        if (sh.np == 1) return (const void*)estep_adjoint_kernel<1, QB, 32, 16, false>;
        if (sh.g <= 4) return (const void*)estep_adjoint_kernel<2, QB, 128, 3, false>;
        return (const void*)estep_adjoint_kernel<2, QB, 256, 1, false>;
    }
    if (sh.np == 1) return (const void*)estep_adjoint_kernel<1, QB, 32, 16, true>;
    if (sh.g <= 4) return (const void*)estep_adjoint_kernel<2, QB, 128, 2, true>;
    return (const void*)estep_adjoint_kernel<2, QB, 256, 1, true>;
}
int occupancy(const void* fn, int threads, size_t smem) {
    int occ = 1;
    cudaFuncSetAttribute(fn, cudaFuncAttributePreferredSharedMemoryCarveout, cudaSharedmemCarveoutMaxShared);
    cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, PPC_MAX * 32);
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, fn, threads, smem) != cudaSuccess || occ < 1) {
        cudaGetLastError();
        occ = 1;
    }
    return occ;
}

}  // namespace

// As many CTAs as fit on the SMs (points of a CTA staged in shared memory, at most PPC_MAX).
int adjoint_grid(int64_t n, int k, bool grad, int num_sms, int64_t* pts_per_cta) {
    const Shape sh = shape_for(k);
    const int occ = occupancy(kernel_for(sh, grad), sh.threads, PPC_MAX / 4 * 32);
    int64_t grid = std::max<int64_t>(1, std::min<int64_t>((n + QB - 1) / QB, (int64_t)num_sms * occ));
    int64_t ppc = ((n + grid - 1) / grid + QB - 1) / QB * QB;
    ppc = std::min<int64_t>(ppc, PPC_MAX);
    grid = (n + ppc - 1) / ppc;
    *pts_per_cta = ppc;
    return (int)grid;
}

int adjoint_class(int k) { return shape_for(k).threads; }

int64_t adjoint_class_points(int k, int64_t points, int num_sms) {
    const Shape sh = shape_for(k);
    const int occ = occupancy(kernel_for(sh, true), sh.threads, 1024 * 32);
    const int64_t ppc = (points + 2LL * num_sms * occ - 1) / (2LL * num_sms * occ);
    return std::min<int64_t>(PPC_MAX, std::max<int64_t>(4 * QB, (ppc + QB - 1) / QB * QB));
}

cudaError_t launch_estep_adjoint(const AdjointLaunch& a, bool grad, int grid, int k_class, cudaStream_t s) {
    const Shape sh = shape_for(k_class);
    void* args[] = {(void*)&a};
    const void* fn = kernel_for(sh, grad);
    note_estep_kernel(fn);
    const size_t smem = (size_t)a.pts_per_cta * 32;
    cudaError_t e = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    return cudaLaunchKernel(fn, dim3(grid), dim3(sh.threads), args, smem, s);
}

int adjoint_components_per_block() { return FIN_CPB; }

cudaError_t launch_adjoint_finalize(const AdjointFinArgs& f, const BatchInst* insts, const int2* blocks, int nblocks,
                                    DeviceState* states, cudaStream_t s) {
    if (insts) grad_finalize_batched_kernel<<<nblocks, FIN_THREADS, 0, s>>>(f, insts, blocks, states);
    else grad_finalize_kernel<<<(f.k + FIN_CPB - 1) / FIN_CPB, FIN_THREADS, 0, s>>>(f);
    return cudaGetLastError();
}

}  // namespace gira
