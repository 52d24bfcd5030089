// gira_internal.cuh -- shared definitions of the libgira CUDA kernels (sm_103a).
//
// Layout of the per-component E-step parameters ("pair-interleaved"):
// components 2p and 2p+1 form pair p; pair p owns PAIR_FLOATS floats at
// params[p * PAIR_FLOATS], stored as float2 slots {comp 2p, comp 2p+1}:
//   slot 0..5   P' = alpha * L^{-1}, lower triangle (p00, p10, p11, p20, p21, p22)
//   slot 6..8   b' = -P' mu
//   slot 9      c  = log2 pi + sum_j log2 (L^{-1})_jj - (3/2) log2(2 pi)
//   slot 10..12 -mu (binary32; mu is also the shift of the M-step statistics)
//   slot 13     the weight behind c: N_b after an M-step (c then uses log2 N_b and
//               the E-step subtracts log2 sum_a N_a), or the caller's weight
//   slot 14     a lower bound of sigma_min(P')^2 = alpha^2 / lambda_max(Sigma): the
//               point-stationary E-step's reach test (a pair whose q' is > 126 over a
//               warp's box of points gives exact zeros and is skipped)
//   slot 15..17 padding: a pair owns 36 floats (144 bytes), so lanes reading the
//               same slot of consecutive pairs in shared memory hit different banks
// alpha = sqrt(log2(e) / 2), so that c - ||P' x + b'||^2 = log2(pi N(x|mu,Sigma))
// (Eq. simplifiedGaussian scaled to base 2).  Padding components carry
// c = -inf, P' = b' = mu = 0, so they contribute exactly zero.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include "gira.h"

namespace gira {

constexpr int PAIR_FLOATS = 36;
constexpr int PAIR_F4 = PAIR_FLOATS / 4;   // float4 per pair block
constexpr int SLOT_P = 0, SLOT_B = 6, SLOT_C = 9, SLOT_NMU = 10, SLOT_W = 13, SLOT_S = 14;
constexpr int NSTAT = 10;   // S0, S1[3], S2[6] (00,01,02,11,12,22)
constexpr int MODEL = 10;   // w, mu[3], Sigma[6] (00,01,02,11,12,22), binary64; w = N_b or caller weight

// Device-side state of one library call (zeroed by the host at call start).
struct DeviceState {
    int error;             // first device-side gira_status (atomicCAS from 0)
    int bad_component;     // component behind GIRA_ERR_NOT_PD
    int stop_after;        // EM: last iteration to run (set on convergence); host sets it to iters
    int iters_done;        // EM iterations completed
    int lloyd_done;        // Lloyd centre updates made
    int w_raw;             // 1 once an M-step has run: weights are N_b, normalised by sum_a N_a on use
    double prev_ll;        // l_{t-1}
    double ll_sum;         // sum_n lse_n of the last E-step (natural log)
    int64_t chosen_last;   // k-means++: index chosen by the last select step
    // point-stationary E-step with statistics, summed over its launches: warp x pair
    // evaluations made (pairs within reach of the warp's box) and with statistics
    unsigned long long pairs_near, pairs_live;
    int coherent;          // k-means++: the points' order keeps neighbours together (launch_kpp_coherence)
    int cmax_ord;          // given models: max_b c_b as an order-preserving int (host: that of -inf)
};
constexpr int CMAX_ORD_NONE = (int)0x807fffff;   // -inf

__device__ __forceinline__ void set_error(DeviceState* st, int code) { atomicCAS(&st->error, 0, code); }

// Raise st->cmax_ord to the largest c of a warp's lanes (-inf: none).  Called by whole warps.
__device__ __forceinline__ void raise_cmax(DeviceState* st, float c) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) c = fmaxf(c, __shfl_xor_sync(0xffffffffu, c, o));
    const int b = __float_as_int(c);
    if ((threadIdx.x & 31) == 0) atomicMax(&st->cmax_ord, b >= 0 ? b : b ^ 0x7fffffff);
}

// Index checks of the debug build (-DGIRA_DEBUG): GIRA_IN(cond, st) is cond, and a
// false cond records GIRA_ERR_BOUNDS in st (the caller skips the access).  In
// release builds it is true and the condition is not evaluated.
#ifdef GIRA_DEBUG
__device__ __forceinline__ bool gira_in(bool ok, DeviceState* st) {
    if (!ok && st) set_error(st, GIRA_ERR_BOUNDS);
    return ok;
}
#define GIRA_IN(cond, st) ::gira::gira_in((cond), (st))
#else
#define GIRA_IN(cond, st) true
#endif

// ---------------------------------------------------------------- packed FP32
__device__ __forceinline__ float2 f2(float a, float b) { return make_float2(a, b); }
__device__ __forceinline__ float2 dup(float a) { return make_float2(a, a); }
__device__ __forceinline__ float2 fma2(float2 a, float2 b, float2 c) { return __ffma2_rn(a, b, c); }
__device__ __forceinline__ float2 add2(float2 a, float2 b) { return __fadd2_rn(a, b); }
__device__ __forceinline__ float2 mul2(float2 a, float2 b) { return __fmul2_rn(a, b); }

// a * b rounded on its own: ptxas contracts a packed multiplication whose result is added
// (__fmul2_rn, and mul.rn.f32x2 too: a probe against the scalar _rn form differed in 21 % of
// random squared distances) and folds an fma with a literal -0; with a -0 it cannot see
// (nz = (-0, -0), a kernel argument) the product stays one rounded operation.  4-D Lloyd uses it;
// the packed 3-D kernels do not (dist2_f32 says what that means).
__device__ __forceinline__ float2 mul2_alone(float2 a, float2 b, float2 nz) { return fma2(a, b, nz); }

__device__ __forceinline__ float ex2_approx(float x) {
    float y;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}
__device__ __forceinline__ float lg2_approx(float x) {
    float y;
    asm("lg2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}

// ---------------------------------------------------------------- warp reductions
struct AddOp {
    __device__ __forceinline__ float operator()(float a, float b) const { return a + b; }
};
struct MaxOp {
    __device__ __forceinline__ float operator()(float a, float b) const { return fmaxf(a, b); }
};

// Per-lane batch index owned after the transpose-reduce: Q = 8 -> bits 4..2 of
// the lane, Q = 4 -> bits 4..3.  The owner of index q is lane q * (32 / Q).
template <int Q>
__device__ __forceinline__ int q_of_lane(int lane) {
    return Q == 8 ? (lane >> 2) & 7 : (lane >> 3) & 3;
}

// Combine Q per-lane values over the 32 lanes of a warp.  On return, lane l
// holds the combination for index q_of_lane<Q>(l); the order of combination is
// fixed, and the lanes sharing an index hold bit-identical results.
template <int Q, class Op>
__device__ __forceinline__ float warp_transpose_reduce(const float (&v)[Q], int lane, Op op) {
    const bool b4 = lane & 16, b3 = lane & 8, b2 = lane & 4;
    float w[Q / 2];
#pragma unroll
    for (int i = 0; i < Q / 2; ++i) {
        const float send = b4 ? v[i] : v[i + Q / 2];
        const float keep = b4 ? v[i + Q / 2] : v[i];
        w[i] = op(keep, __shfl_xor_sync(0xffffffffu, send, 16));
    }
    float t;
    if (Q == 8) {
        float z[2];
#pragma unroll
        for (int i = 0; i < 2; ++i) {
            const float send = b3 ? w[i] : w[i + 2];
            const float keep = b3 ? w[i + 2] : w[i];
            z[i] = op(keep, __shfl_xor_sync(0xffffffffu, send, 8));
        }
        const float send = b2 ? z[0] : z[1];
        const float keep = b2 ? z[1] : z[0];
        t = op(keep, __shfl_xor_sync(0xffffffffu, send, 4));
    } else {
        const float send = b3 ? w[0] : w[1];
        const float keep = b3 ? w[1] : w[0];
        t = op(keep, __shfl_xor_sync(0xffffffffu, send, 8));
        t = op(t, __shfl_xor_sync(0xffffffffu, t, 4));
    }
    t = op(t, __shfl_xor_sync(0xffffffffu, t, 2));
    t = op(t, __shfl_xor_sync(0xffffffffu, t, 1));
    return t;
}


// ---------------------------------------------------------------- TMA bulk copy + mbarrier
// (PTX ISA: cp.async.bulk, mbarrier; a plain launch is a cluster of one CTA, so
// the CTA's own shared memory is addressed through the shared::cluster window.)
__device__ __forceinline__ uint32_t smem_u32(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }

__device__ __forceinline__ void mbar_init(uint64_t* bar, uint32_t count) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(bar)), "r"(count) : "memory");
}
__device__ __forceinline__ void mbar_fence_init() { asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory"); }
__device__ __forceinline__ void mbar_expect_tx(uint64_t* bar, uint32_t bytes) {
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(bar)), "r"(bytes) : "memory");
}
// bytes: multiple of 16; src and dst 16-byte aligned.
__device__ __forceinline__ void tma_load_1d(void* dst, const void* src, uint32_t bytes, uint64_t* bar) {
    asm volatile(
        "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(smem_u32(dst)),
        "l"(src), "r"(bytes), "r"(smem_u32(bar))
        : "memory");
}
__device__ __forceinline__ bool mbar_try_wait(uint64_t* bar, uint32_t parity) {
    uint32_t ok;
    asm volatile(
        "{\n\t.reg .pred p;\n\tmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\tselp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(ok)
        : "r"(smem_u32(bar)), "r"(parity)
        : "memory");
    return ok != 0;
}
// Programmatic dependent launch (PTX griddepcontrol).  In a kernel launched with
// programmatic stream serialisation, pdl_wait() returns once the previous kernel
// of the stream has completed and its writes are visible, and pdl_allow_next()
// lets the next such kernel be scheduled before this one ends.  In a plain
// launch both have no effect.
__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void pdl_allow_next() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
__device__ __forceinline__ uint64_t globaltimer_ns() {
    uint64_t t;
    asm volatile("mov.u64 %0, %globaltimer;" : "=l"(t));
    return t;
}
// Bounded wait for the phase with the given parity: false once `limit_ns` of
// wall time has passed (try_wait itself may suspend between polls).
__device__ __forceinline__ bool mbar_wait_bounded(uint64_t* bar, uint32_t parity, long long limit_ns) {
    if (mbar_try_wait(bar, parity)) return true;
    const uint64_t t0 = globaltimer_ns();
    while (true) {
        if (mbar_try_wait(bar, parity)) return true;
        if (globaltimer_ns() - t0 > (uint64_t)limit_ns) return false;
    }
}

// ---------------------------------------------------------------- bounded waits on global memory
__device__ __forceinline__ int ld_acquire(const int* p) {
    int v;
    asm volatile("ld.acquire.gpu.global.s32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
    return v;
}
__device__ __forceinline__ void st_release(int* p, int v) {
    asm volatile("st.release.gpu.global.s32 [%0], %1;" ::"l"(p), "r"(v) : "memory");
}
// Wait until *counter >= target.  false when *abort is raised by another waiter,
// or after `limit` polls (each followed by a short sleep): then this waiter
// records GIRA_ERR_TIMEOUT and raises *abort so that the others leave too.
__device__ __forceinline__ bool wait_counter_bounded(const int* counter, int target, int* abort, long long limit,
                                                     DeviceState* st) {
    long long spins = 0;
    while (ld_acquire(counter) < target) {
        if (ld_acquire(abort)) return false;
        if (++spins > limit) {
            set_error(st, GIRA_ERR_TIMEOUT);
            st_release(abort, 1);
            return false;
        }
        __nanosleep(32);
    }
    return true;
}

// binary32 squared distance in the fixed order d_i = x_i - c_i; (d0^2 + d1^2) + d2^2,
// every operation rounded separately (no contraction): the D^2 of the seeding kernels over
// sub-blocks, of the persistent one and of two launches per centre, and (dist2_f32_4) every
// distance in four dimensions.  The packed 3-D kernels (kpp_cluster_kernel and Lloyd's
// assignment) write the same order, but the compiler fuses the additions with the products: they
// compute fma(d2, d2, fma(d0, d0, d1^2)) (the labels of 156,000 near ties are that form's, every
// one), within 1.5 units in the last place of it.  Labels then differ from this arithmetic's only
// between centres whose distances agree to 2^-22 (about one point in a few frames), draws only
// where the running sum meets the threshold within that rounding (none in 26 seedings of 100 to
// 512 centres compared).
__device__ __forceinline__ float dist2_f32(float4 x, float4 c) {
    float d0 = __fsub_rn(x.x, c.x), d1 = __fsub_rn(x.y, c.y), d2 = __fsub_rn(x.z, c.z);
    float s = __fadd_rn(__fmul_rn(d0, d0), __fmul_rn(d1, d1));
    return __fadd_rn(s, __fmul_rn(d2, d2));
}
// Four dimensions: ((d0^2 + d1^2) + d2^2) + d3^2, same rules.
__device__ __forceinline__ float dist2_f32_4(float4 x, float4 c) {
    const float d3 = __fsub_rn(x.w, c.w);
    return __fadd_rn(dist2_f32(x, c), __fmul_rn(d3, d3));
}

// ---------------------------------------------------------------- exact fixed-point weights
// k-means++ weights: fx(d) = floor(d * 2^48) for a binary32 d >= 0 (saturating
// at 2^95 - 1 for d >= 2^47), summed exactly in 128 bits; the draw threshold is
// floor(k * T / 2^53) for the 53-bit integer k behind u and the total T.
struct u128 {
    unsigned long long lo, hi;
};
__host__ __device__ __forceinline__ u128 u128_add(u128 a, u128 b) {
    u128 r;
    r.lo = a.lo + b.lo;
    r.hi = a.hi + b.hi + (r.lo < a.lo ? 1ull : 0ull);
    return r;
}
__host__ __device__ __forceinline__ u128 u128_sub(u128 a, u128 b) {
    u128 r;
    r.lo = a.lo - b.lo;
    r.hi = a.hi - b.hi - (a.lo < b.lo ? 1ull : 0ull);
    return r;
}
__host__ __device__ __forceinline__ bool u128_gt(u128 a, u128 b) { return a.hi > b.hi || (a.hi == b.hi && a.lo > b.lo); }
__host__ __device__ __forceinline__ bool u128_zero(u128 a) { return (a.lo | a.hi) == 0ull; }
__device__ __forceinline__ u128 u128_shfl_up(u128 v, int o) {
    u128 r;
    r.lo = __shfl_up_sync(0xffffffffu, v.lo, o);
    r.hi = __shfl_up_sync(0xffffffffu, v.hi, o);
    return r;
}
__device__ __forceinline__ u128 u128_shfl(u128 v, int src) {
    u128 r;
    r.lo = __shfl_sync(0xffffffffu, v.lo, src);
    r.hi = __shfl_sync(0xffffffffu, v.hi, src);
    return r;
}
// Inclusive warp scan (exact, so the order of the additions does not matter).
__device__ __forceinline__ u128 u128_warp_incl_scan(u128 v, int lane) {
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const u128 u = u128_shfl_up(v, o);
        if (lane >= o) v = u128_add(v, u);
    }
    return v;
}
__device__ __forceinline__ u128 fx48(float d) {
    u128 r{0ull, 0ull};
    if (!(d > 0.f)) return r;
    if (d >= 140737488355328.0f) return u128{~0ull, (1ull << 31) - 1ull};   // 2^47 -> 2^95 - 1
    const unsigned bits = __float_as_uint(d);
    const int ex = (int)(bits >> 23);
    const unsigned long long mant = (bits & 0x7FFFFFu) | (ex ? 0x800000u : 0u);
    const int sh = (ex ? ex : 1) - 150 + 48;   // d = mant * 2^(sh - 48)
    if (sh >= 64) {
        r.hi = mant << (sh - 64);
    } else if (sh > 40) {
        r.lo = mant << sh;
        r.hi = mant >> (64 - sh);
    } else if (sh >= 0) {
        r.lo = mant << sh;
    } else if (sh > -24) {
        r.lo = mant >> (-sh);
    }
    return r;
}
__device__ __forceinline__ u128 fx_threshold(unsigned long long k53, u128 T) {
    const unsigned long long a_lo = k53 * T.lo, a_hi = __umul64hi(k53, T.lo);
    const unsigned long long b_lo = k53 * T.hi, b_hi = __umul64hi(k53, T.hi);
    const unsigned long long w0 = a_lo, w1 = a_hi + b_lo;
    const unsigned long long w2 = b_hi + (w1 < a_hi ? 1ull : 0ull);
    return u128{(w0 >> 53) | (w1 << 11), (w1 >> 53) | (w2 << 11)};
}

// SplitMix64 (Steele, Lea & Flood 2014) as a counter-based generator:
// draw j of `seed` is output j+1 of the stream started at state `seed`.
__host__ __device__ __forceinline__ uint64_t splitmix64(uint64_t seed, uint64_t j) {
    uint64_t z = seed + (j + 1) * 0x9E3779B97F4A7C15ull;
    z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
    z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
    return z ^ (z >> 31);
}
__host__ __device__ __forceinline__ double uniform53(uint64_t seed, uint64_t j) {
    return (double)(splitmix64(seed, j) >> 11) * (1.0 / 9007199254740992.0);
}

// K above this runs the E-step over reach lists (reach_kernels.cu); the batched and
// no-allocation entry points take K up to it only.
constexpr int MAX_K_DIRECT = 1024;

// ---------------------------------------------------------------- kernel entry points
// (defined in em_kernels.cu / kmeans_kernels.cu, launched from gira_api.cu)

// Runs of equal keys over a warp whose lanes hold consecutive elements: a lane has key_first ..
// key_last with the sum and count of its last run and, unless it is `whole` (one run), of its
// first.  Runs that go on over lanes are joined by a segmented scan of the lanes' last runs
// (fixed order) and put(key, sum, count) is called once for each.  Called by whole warps.
template <int NV, class Put>
__device__ __forceinline__ void join_runs(int key_first, int key_last, bool whole, double (&first)[NV], int nfirst,
                                          double (&run)[NV], int nrun, Put put) {
    constexpr unsigned ALL = 0xffffffffu;
    const int lane = threadIdx.x & 31;
    const int before = __shfl_up_sync(ALL, key_last, 1), after = __shfl_down_sync(ALL, key_first, 1);
    const bool joins = lane > 0 && before == key_first;   // the lane's first run goes on from the lane before
    const unsigned heads = __ballot_sync(ALL, !(whole && joins));
    const int start = 31 - __clz(heads & (ALL >> (31 - lane)));
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        if (__all_sync(ALL, lane - o < start)) break;   // no run is longer
        const int c = __shfl_up_sync(ALL, nrun, o);
        if (lane - o >= start) nrun += c;
#pragma unroll
        for (int q = 0; q < NV; ++q) {
            const double u = __shfl_up_sync(ALL, run[q], o);
            if (lane - o >= start) run[q] += u;
        }
    }
    const int nprev = __shfl_up_sync(ALL, nrun, 1);
#pragma unroll
    for (int q = 0; q < NV; ++q) {
        const double u = __shfl_up_sync(ALL, run[q], 1);
        if (!whole && joins) first[q] += u;
    }
    if (!whole) put(key_first, first, nfirst + (joins ? nprev : 0));
    if (lane == 31 || after != key_last) put(key_last, run, nrun);
}

// sums[(D + 1) key + q] += the coordinates (binary64) and the count of a warp's 128 points, lane l
// holding points 4 l .. 4 l + 3 with labels key[0 .. 3] (-1: none, only at the end).  Runs of equal
// labels are summed first, inside the lane and then over the lanes (a segmented scan of the lanes'
// last runs, fixed order), so that neighbours cost few atomics -- and few binary64 instructions,
// which bound this (64 cycles each per warp): 39 for 128 points in 3-D, where one point per lane
// and a scan for each of four rounds took 92.
// Points in no order under two to four labels have dozens of runs a warp and all their atomics
// on a few addresses: there (CROWDED: up to four labels in all, more than 4,096 points) each label's
// points are summed over the warp instead, in a fixed order, for one set of atomics each.  KInit with
// five Lloyd iterations of shuffled points, K = 2: 300,000 2,750 us by runs, 335 so; 20,000 341 and 170;
// but 1,000 139 and 169.
constexpr int CROWDED_LABELS = 4, CROWDED_POINTS = 4096;
template <int D, bool CROWDED>
__device__ __forceinline__ void add_runs(const int (&key)[4], const float (&x)[4][D], double* sums) {
    auto put = [&](int k, const double (&v)[D], int c) {
        if (k < 0) return;
        double* s = sums + (size_t)(D + 1) * k;
#pragma unroll
        for (int q = 0; q < D; ++q) atomicAdd(s + q, v[q]);
        atomicAdd(s + D, (double)c);
    };
    constexpr unsigned ALL = 0xffffffffu;
    constexpr int MANY = 24, LABELS = CROWDED_LABELS + 1;   // and -1
    if (CROWDED && __reduce_add_sync(ALL, (key[1] != key[0]) + (key[2] != key[1]) + (key[3] != key[2])) >= MANY) {
        int label[LABELS], found = 0;
        unsigned open = 0xfu;   // this lane's points whose label is not found yet
#pragma unroll
        for (int t = 0; t < LABELS; ++t) {
            label[t] = -1;
            const unsigned lanes = __ballot_sync(ALL, open != 0u);
            if (lanes == 0u) continue;
            const int mine = key[open ? __ffs(open) - 1 : 0];
            label[t] = __shfl_sync(ALL, mine, __ffs(lanes) - 1);
            found = t + 1;
#pragma unroll
            for (int r = 0; r < 4; ++r)
                if (key[r] == label[t]) open &= ~(1u << r);
        }
        if (!__any_sync(ALL, open != 0u)) {
            for (int t = 0; t < found; ++t) {
                double v[D];
                int c = 0;
#pragma unroll
                for (int q = 0; q < D; ++q) v[q] = 0.0;
#pragma unroll
                for (int r = 0; r < 4; ++r)
                    if (key[r] == label[t]) {
                        ++c;
#pragma unroll
                        for (int q = 0; q < D; ++q) v[q] += (double)x[r][q];
                    }
                c = __reduce_add_sync(ALL, c);
#pragma unroll
                for (int q = 0; q < D; ++q)
#pragma unroll
                    for (int o = 16; o > 0; o >>= 1) v[q] += __shfl_xor_sync(ALL, v[q], o);
                if ((threadIdx.x & 31) == 0) put(label[t], v, c);
            }
            return;
        }
    }
    double run[D], first[D];   // the lane's last run and, when it has several, its first
    int nrun = 1, nfirst = 0;
    bool whole = true;
#pragma unroll
    for (int q = 0; q < D; ++q) {
        run[q] = (double)x[0][q];
        first[q] = 0.0;
    }
#pragma unroll
    for (int r = 1; r < 4; ++r) {
        if (key[r] == key[r - 1]) {
#pragma unroll
            for (int q = 0; q < D; ++q) run[q] += (double)x[r][q];
            ++nrun;
        } else {
            if (whole) {
#pragma unroll
                for (int q = 0; q < D; ++q) first[q] = run[q];
                nfirst = nrun;
                whole = false;
            } else {
                put(key[r - 1], run, nrun);
            }
#pragma unroll
            for (int q = 0; q < D; ++q) run[q] = (double)x[r][q];
            nrun = 1;
        }
    }
    join_runs(key[0], key[3], whole, first, nfirst, run, nrun, put);
}

// Batched fits: one entry per instance (device table).
struct BatchInst {
    int64_t pt_off;     // first point of the instance in the packed point arrays
    int64_t n;          // its points
    int64_t ppc;        // points per E-step CTA
    int64_t par_off;    // float offset of its E-step parameters (its class's padded pair count)
    int64_t part_off;   // float offset of its per-CTA statistic partials ([ctas][k][NSTAT])
    int64_t ll_off;     // double offset of its per-CTA log-likelihood partials
    int k;              // components
    int comp_off;       // first component in the per-component arrays
    int ctas;           // E-step CTAs of the instance
    int pad_;
    int64_t mask_off;   // word offset of its live masks
    int64_t live_off;   // word offset of its live-slice masks (gradient)
};
// One E-step CTA of a batched launch: instance and CTA index within it.
struct BatchUnit {
    int inst, cta;
};

// Slices of the statistics over n points, of *sr blocks of 128 points each: the unit of
// work is one (slice, pair).  8 blocks (in Morton order a pair's live blocks lie in a few
// slices, and longer ones leave few, long units), more above 512 slices, which bounds the
// partial rows.
__host__ __device__ inline int reach_slices(int64_t n, int* sr) {
    const int64_t rows = (n + 127) / 128;
    int r = 8;
    while (rows > 512 * (int64_t)r) r *= 2;
    *sr = r;
    return (int)((rows + r - 1) / r);
}

// The E-step over reach lists (reach_kernels.cu).
struct ReachLaunch {
    const float4* pts8;      // 2 float4 per point, as EStepLaunch (4-D: (x,x,y,y) (z,z,I,I))
    int64_t n;
    int k;
    const float* params;     // pair-interleaved
    const float4* ctr;       // compact per-component arrays and references of launch_reach_prepare,
                             // or the arrays of the launch that built a given model
    const float2* aux;
    const float* gref;       // nullptr (given models): max_b c_b from st->cmax_ord
    double* llp;             // [grid] log-likelihood partials
    float* per_point;        // mode 0: [n] natural-log lse, or nullptr
    DeviceState* st;
    int iter;
    int64_t n_buf = 0;       // points in pts8 (index checks of the debug build; 0: unchecked)
    float2* pref = nullptr;  // [n] (shift, 1 / total): with masks
    uint32_t* masks = nullptr;   // [reach_mask_words(k)][rows] live pairs per block of 128 points
    int64_t rows = 0;
    // with masks: the same per slice, [reach_mask_words(k)][slices], and the (slice, pair)s
    // with work: units[0 .. count), count in unit_count[0] ([1]: the statistics' cursor);
    // live2 and unit_count are zeroed before the launch
    uint32_t* live2 = nullptr;
    uint2* stat_units = nullptr;   // (instance, slice << 16 | pair)
    int* unit_count = nullptr;
    // gradient (mode 2)
    float* grad_pts = nullptr;        // [n][3], at order[i] (or i) for the i-th point, or nullptr
    const int* order = nullptr;
    const float* rot = nullptr;       // batch x 12: R (row-major) of x' = R x + t, then t
    double* pose_partials = nullptr;  // [grid][12]
    // batched gradient launches: as EStepLaunch
    const BatchInst* insts = nullptr;
    const BatchUnit* units = nullptr;
    DeviceState* states = nullptr;
};
int reach_h(int64_t n);        // warps per block of 128 points for n points in the launch
int reach_points(int h);       // points per CTA
int reach_grid(int64_t n);     // CTAs of a single launch
int64_t reach_rows(int64_t n); // blocks of 128 points
int reach_mask_words(int k);
cudaError_t launch_reach_prepare(int d, const float* params, int k, const DeviceState* st, int iter, float4* ctr, float2* aux,
                                 float* gref, cudaStream_t s);
// d: 3 or 4 dimensions.  mode 0 log-likelihood, 1 with masks and pref, 2 gradient (3-D); h: reach_h of the launch; kmax: the largest k.
cudaError_t launch_estep_reach(int d, const ReachLaunch& a, int mode, int grid, int h, int kmax, cudaStream_t s);
// partials [slices][pairs][2 NSTAT (4-D: NSTAT4)], written where a.live2 has the bit:
// launch_reduce_finalize takes the two as rows and masks.  world (4-D): about x - mu, not whitened.
cudaError_t launch_reach_stats(int d, const ReachLaunch& a, bool world, float* partials, cudaStream_t s);

struct EStepLaunch {
    const float4* pts8;      // 2 float4 per point: (x,x,y,y) (z,z,0,0)
    int64_t n;
    int k;
    const float* params;     // pair-interleaved, npairs_pad * PAIR_FLOATS
    float* partials;         // statistics (stats launches), see masks
    double* ll_partials;     // [grid]
    float* per_point;        // [n] natural-log lse, or nullptr
    DeviceState* st;
    int iter;                // iteration index (1-based); kernels skip if iter > st->stop_after
    // batched launches: CTA b runs units[b]; pts8 / params / partials / ll_partials /
    // per_point are then bases offset by the instance's table entry, st = states + inst
    const BatchInst* insts = nullptr;
    const BatchUnit* units = nullptr;
    DeviceState* states = nullptr;
    // point-stationary E-step (estep_pt_kernel): partial rows [rows][pairs][2 NSTAT],
    // row cta * PT_B + block written only where the block's live mask has the pair's
    // bit, and the live masks [npairs / 32][rows] (bit p: pair p reaches some point
    // of the block)
    uint32_t* masks = nullptr;
    int64_t pt_rows = 0;   // point blocks of the launch (the row count of partials and masks)
    int64_t n_buf = 0;     // points in pts8 (index checks of the debug build; 0: unchecked)
    // CTA order of a single fit's E-step: from iteration 3 on, CTA blockIdx.x takes the
    // point blocks of CTA cta_perm[(iter & 1) * grid + blockIdx.x] (longest expected
    // work first, written by the finalize two iterations earlier); cta_key[cta]
    // receives the CTA's work key for that order (nullptr: launch order, no keys)
    const int* cta_perm = nullptr;
    uint8_t* cta_key = nullptr;
};

// A launch configuration, with programmatic stream serialisation when pdl (the
// kernel may start before the previous kernel in the stream has finished, and
// waits for it with pdl_wait()).
struct PdlConfig {
    cudaLaunchConfig_t cfg{};
    cudaLaunchAttribute at[1];
    PdlConfig(dim3 grid, dim3 block, size_t smem, cudaStream_t s, bool pdl) {
        cfg.gridDim = grid;
        cfg.blockDim = block;
        cfg.dynamicSmemBytes = smem;
        cfg.stream = s;
        at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
        at[0].val.programmaticStreamSerializationAllowed = 1;
        cfg.attrs = at;
        cfg.numAttrs = pdl ? 1 : 0;
    }
};
// Pairs (padded) the parameter buffer must hold for k components.
int params_pairs_padded(int k);

// N x 3 -> pts4 (x,y,z,0) (nullable) and pts8 (x,x,y,y)(z,z,0,0); flags non-finite input.
cudaError_t launch_pack(const float* pts3, int64_t n, float4* pts4, float4* pts8, DeviceState* st, cudaStream_t s);
// Spatial order of packed points (order_kernels.cu): a stable radix sort by
// (instance, 18-bit Morton code in the instance's bounding cube).  offsets_d /
// units_d: the batch's point offsets and its (instance, chunk) bounding-box
// blocks (point_order_fill_units), or nullptr for one instance of n points.
// Writes the sorted points to p8_out (and, if p4_out, as (x, y, z, 0)) and, if
// order_out, the source index of every sorted point.  scratch: point_order_scratch_bytes(n, batch) bytes.
int64_t point_order_box_units(const int64_t* offsets, int batch);
void point_order_fill_units(const int64_t* offsets, int batch, int2* units);
size_t point_order_scratch_bytes(int64_t n, int batch);
int point_order_launches(int batch);   // kernels one launch_point_order makes
int64_t point_order_max_n();          // larger inputs keep the caller's order
cudaError_t launch_point_order(const float4* p8, int64_t n, const int64_t* offsets_d, const int2* units_d,
                               int nunits, int batch, void* scratch, float4* p8_out, float4* p4_out, int* order_out,
                               cudaStream_t s);
// The points of an n x 3 array cell by cell (a 32^3 grid over their bounding box, cells in
// Morton order, no fixed order inside a cell): order.  For kernels whose result per point
// does not depend on the order.  scratch: cell_group_scratch_bytes(n) bytes, n < 2^31.
size_t cell_group_scratch_bytes(int64_t n);
int cell_group_launches();
cudaError_t launch_cell_group(const float* p3, int64_t n, void* scratch, int* order, cudaStream_t s);
cudaError_t launch_fill_padding(float* params, int k, int npairs_pad, cudaStream_t s);
// Sum of the per-CTA log-likelihoods into st->ll_sum (fixed order).
cudaError_t launch_ll_reduce(const double* ll_partials, int grid, DeviceState* st, cudaStream_t s);
// M-step: reduce the per-CTA partials (or read binary64 stats64 when partials is
// nullptr), then binary64 finalize of every component; EM iterations (em) also
// reduce the log-likelihood, write the trace and decide convergence.
cudaError_t launch_reduce_finalize(const float* partials, int grid, const double* ll_partials,
                                   const double* stats64, float4* shift4, int k, int64_t n, double reg, double tol,
                                   double* model64, float* params, double* trace, DeviceState* st, int iter, bool em,
                                   cudaStream_t s, bool pdl = false, const int* perm = nullptr,
                                   const uint32_t* masks = nullptr, int nwords = 0, int ll_count = 0,
                                   const uint8_t* cta_key = nullptr, int* cta_perm = nullptr, int cta_grid = 0);
// Point-stationary E-step (3-D fits and log-likelihood, k <= 1024): CTAs for n
// points; partial rows (warps) of a grid; live-mask words per warp for k.
int estep_pt_grid(int64_t n);
int estep_pt_rows(int grid);
int estep_pt_row_floats(int k);   // floats of one partial row of the point-stationary E-step
int estep_pt_mask_words(int k);
// a.partials: [k * NSTAT][rows] (stats), a.masks: [mask words][rows], a.pt_rows = rows,
// a.ll_partials: [grid]
cudaError_t launch_estep_pt(const EStepLaunch& a, bool stats, int grid, cudaStream_t s, bool pdl = false);
// The same over a unit table (batched fits; a.insts / a.units / a.states; every
// instance's part_off, mask_off, ll_off and ctas for PT points per CTA).
cudaError_t launch_estep_pt_units(const EStepLaunch& a, bool stats, int nunits, int kmax, cudaStream_t s);
int estep_pt_points();   // points per CTA
int estep_pt_blocks();   // point blocks per CTA (partial and mask rows per CTA)
// ctr, aux (nullable): the compact arrays of the reach tests, and max_b c_b in st->cmax_ord.
cudaError_t launch_model_points(const float* pts3, int64_t n, float4* pts8, const float* w, const float* mu,
                                const float* cov, int k, int npairs_pad, double* model64, float* params,
                                float4* shift4, float4* ctr, float2* aux, DeviceState* st, cudaStream_t s);
// perm (nullable): slot s of model64 is the caller's component perm[s].
cudaError_t launch_model_out(const double* model64, int k, float* w, float* mu, float* cov, const DeviceState* st,
                             cudaStream_t s, const int* perm = nullptr);
// Morton order of the k <= 8192 means at old[b * stride + 1 ..] (rows of a binary64 model): perm.
cudaError_t launch_order_means(const double* old, int stride, int k, int* perm, cudaStream_t s);
// Reorder the k <= 8192 components of model64 along a space-filling curve of
// their means (Morton order) and rebuild params / shift4 / model64 in that order:
// slot s holds the caller's component perm[s].  scratch: k * MODEL doubles.
cudaError_t launch_order_components(double* model64, double* scratch, int k, int* perm, float* params,
                                    float4* shift4, DeviceState* st, cudaStream_t s);

// Batched EM (per-instance tables on the device).
cudaError_t launch_pack_batched(const float* pts3, int64_t n, const int64_t* offsets, int batch, float4* pts4,
                                float4* pts8, DeviceState* states, cudaStream_t s);
// Finalize blocks: (instance, block index within the instance), FIN_CPB components each.
int fin_components_per_block();
// stats64: the one-hot statistics (partials == nullptr), or room for the sums; comp_inst: the
// instance of each of the total_k components.  Large batches take two launches
// (finalize_batched_splits) when there are partials.
bool finalize_batched_splits(int nblocks);
cudaError_t launch_reduce_finalize_batched(const float* partials, const double* ll_partials, double* stats64,
                                           float4* shift4, const BatchInst* insts, const int2* blocks, int nblocks,
                                           const int* comp_inst, int total_k, double reg, double tol, int iters,
                                           double* model64, float* params, double* trace, DeviceState* states,
                                           int iter, bool em, cudaStream_t s, const int* perm = nullptr,
                                           const uint32_t* masks = nullptr);
// Padding slots of every instance's parameter block (one block per instance).
cudaError_t launch_fill_padding_batched(float* params, const BatchInst* insts, int batch, int npairs_max,
                                        const int* npairs_of, cudaStream_t s);
// E-step parameters of every instance from (w, mu, Sigma) (comp_inst: instance of each component).
cudaError_t launch_params_from_model_batched(const float* w, const float* mu, const float* cov, int total_k,
                                             const int* comp_inst, const BatchInst* insts, double* model64,
                                             float* params, float4* shift4, DeviceState* states, cudaStream_t s);
// Normalised model of every instance (one block per instance).
cudaError_t launch_model_out_batched(const double* model64, const BatchInst* insts, int batch, float* w, float* mu,
                                     float* cov, const DeviceState* states, cudaStream_t s,
                                     const int* perm = nullptr);
// launch_order_components for every instance of a batch (one block each, k <= 8192).
cudaError_t launch_order_components_batched(double* model64, double* scratch, int total_k, int kmax,
                                            const BatchInst* insts, int batch, const int* comp_inst, int* perm,
                                            float* params, float4* shift4, DeviceState* states, cudaStream_t s);
// Per-instance sums of the log-likelihood partials into states[i].ll_sum.
cudaError_t launch_ll_reduce_batched(const double* ll_partials, const BatchInst* insts, int batch,
                                     DeviceState* states, cudaStream_t s);

// Batched differentiable log-likelihood (a batch table of scans, each with its
// own model and pose; poses: batch x 12, or nullptr for identities).
cudaError_t launch_pack_pose_batched(const float* pts3, int64_t n, const int64_t* offsets, int batch,
                                     const float* poses, float4* pts8, DeviceState* states, cudaStream_t s);
// The gradient with every component, statistics in world axes (adjoint_kernels.cu).
struct AdjointLaunch {
    const float4* pts8;      // as EStepLaunch, in the caller's order
    int64_t n;
    int k;
    const float* params;     // in the caller's order, padded to params_pairs_padded(k)
    int64_t pts_per_cta;     // batched: the largest of the launch (its instances' ppc)
    float* partials;         // [grid][k][NSTAT]
    double* ll_partials;     // [grid]
    DeviceState* st;
    int iter;
    float* grad_pts;         // [n][3] dL/dx, or nullptr
    const float* rot;        // R, row-major 3x3, of x' = R x + t; nullptr = identity
    double* pose_partials;   // [grid][12]: per CTA sum dL/dx' x'^T (row-major), sum dL/dx'
    // batched: CTA b runs units[b]; the pointers are bases offset by the instance's entry
    const BatchInst* insts = nullptr;
    const BatchUnit* units = nullptr;
    DeviceState* states = nullptr;
};
struct AdjointFinArgs {
    const float* partials;
    int grid;
    const double* llp;
    const double* pp;
    const float* pose;
    const float* chol;
    const double* model64;
    int k;
    int64_t n;
    float *g_logits, *g_means, *g_chol;
    double *g_pose, *g_twist;
    DeviceState* st;
};
int adjoint_grid(int64_t n, int k, bool grad, int num_sms, int64_t* pts_per_cta);
int adjoint_class(int k);   // instances of equal class run in one launch
int64_t adjoint_class_points(int k, int64_t points, int num_sms);   // points per CTA of a class
// grad = false: the log-likelihood alone.
cudaError_t launch_estep_adjoint(const AdjointLaunch& a, bool grad, int grid, int k_class, cudaStream_t s);
int adjoint_components_per_block();
cudaError_t launch_adjoint_finalize(const AdjointFinArgs& f, const BatchInst* insts, const int2* blocks, int nblocks,
                                    DeviceState* states, cudaStream_t s);

// Differentiable log-likelihood.  pose12 = R (row-major) then t, or nullptr.
// N x 3 -> pts8 of x' = R x + t (binary32, fixed order); flags non-finite input.
cudaError_t launch_pack_pose(const float* pts3, int64_t n, const float* pose12, float4* pts8, DeviceState* st,
                             cudaStream_t s);
// E-step parameters from (logits, means, Cholesky factors), k <= MAX_K_DIRECT, in Morton
// order of the means (perm[slot]: the caller's component), with the compact arrays of the
// reach tests and max_b c_b in st->cmax_ord.  insts: every instance of a batch, kmax the
// largest k (one fit: its k).  perm nullptr: the caller's order (ctr and aux are not written).
cudaError_t launch_params_from_chol(const float* logits, const float* mu, const float* chol, int kmax,
                                    const BatchInst* insts, int batch, double* model64, float* params, float4* shift4,
                                    int* perm, float4* ctr, float2* aux, DeviceState* st, cudaStream_t s);
// Sums of a gradient launch (fixed order): dL/dlogits (k), dL/dmeans (k x 3) in binary32
// from the statistics, in the caller's order; in binary64 dL/dpose (dL/dR row-major, dL/dt) and dL/dtwist (omega, v); the log-likelihood in
// st->ll_sum, for every instance of a batch (bases offset by its table entry).
// partials nullptr: no parameter gradients.
struct ReachGradArgs {
    const float* partials;    // [slices][pairs][2 NSTAT], live where live2 says
    const uint32_t* live2;    // [words][slices]
    const double* llp;        // per CTA
    const double* pp;         // per CTA, 12 each
    const float* poses;       // batch x 12
    const float* params;
    const double* model64;
    const int* perm;
    int kmax;                 // the largest k
    float *g_logits, *g_means;
    double *g_pose, *g_twist;
    DeviceState* states;
};
cudaError_t launch_reach_grad_finalize(const ReachGradArgs& f, const BatchInst* insts, int batch, cudaStream_t s);

// k-means
// dim: 3 (distances over x, y, z) or 4 (also the fourth coordinate)
cudaError_t launch_kpp(const float4* pts4, int64_t n, int k, uint64_t seed, float4* centers, float* d2,
                       u128* blocksums, int64_t* chosen, DeviceState* st, cudaStream_t s, int dim = 3);
int kpp_num_blocks(int64_t n);
// Persistent k-means++ (one cooperative launch for all K centres).  Grid size, or
// 0 when cooperative launch is unavailable (the per-centre launches are used).
int kpp_persistent_grid();
// sync_ints: k+1 zeroed ints (per-centre arrival counters, abort flag);
// sums: kpp_persistent_sum_words(grid, k) 128-bit words; d2: 2n floats.  Valid for
// n <= kpp_persistent_max_n(grid) (points held in registers).
size_t kpp_persistent_sum_words(int grid, int k);
int64_t kpp_persistent_max_n(int grid);
cudaError_t launch_kpp_persistent(const float4* pts4, int64_t n, int k, uint64_t seed, float4* centers, float* d2,
                                  int64_t* chosen, int* sync_ints, u128* sums, int grid, DeviceState* st,
                                  cudaStream_t s, int dim = 3);
// k-means++ by one cluster over sub-blocks of 32 points kept in L2 (any dim): sub-blocks per
// warp for n points (0: not applicable); worth it when the points' order is coherent
// (launch_kpp_coherence sets st->coherent) or each warp has few.  d2: n floats.
int kpp_blocks_per_warp(int64_t n, int dim);
cudaError_t launch_kpp_coherence(const float4* pts4, int64_t n, int dim, DeviceState* st, cudaStream_t s);
cudaError_t launch_kpp_blocks(const float4* pts4, int64_t n, int k, uint64_t seed, float4* centers, int64_t* chosen,
                              float* d2, int nsb, DeviceState* st, cudaStream_t s, int dim);
// Batched KInit: one entry per instance.
struct KppInst {
    int64_t pt_off, n;
    int k, comp_off, inst, pad_;
};
// Batched seeding: cluster c of the launch (cs CTAs each) seeds instance
// table[c]; every instance needs n <= kpp_cluster_capacity(cs).
cudaError_t launch_kpp_cluster_batched(const float4* pts4, const KppInst* table, int clusters, uint64_t seed,
                                       float4* centers, int64_t* chosen, int cs, DeviceState* states,
                                       cudaStream_t s);
int kpp_cluster_capacity(int cs);
// Batched Lloyd: units (instance, tile of lloyd_tile() points); per-instance
// label / sum / changed slabs (changed: lloyd_iters + 1 counters per instance).
int lloyd_tile();
cudaError_t launch_lloyd_batched(const float4* pts4, const KppInst* table, const BatchUnit* units, int nunits,
                                 int total_k, const int* comp_inst, int lloyd_iters, float4* centers, int32_t* labels,
                                 double* sums, unsigned long long* changed, DeviceState* states, cudaStream_t s);
// One-hot statistics of every instance (instance of point i by binary search over offsets).
cudaError_t launch_label_stats_batched(const float4* pts4, int64_t n, const int64_t* offsets, int batch,
                                       const KppInst* table, const int32_t* labels, const float4* shift4,
                                       double* stats64, DeviceState* states, cudaStream_t s);
// One-cluster k-means++ (no global synchronisation): cluster size for n points,
// or 0 when the one-cluster path does not apply.
int kpp_cluster_size(int64_t n);
cudaError_t launch_kpp_cluster(const float4* pts4, int64_t n, int k, uint64_t seed, float4* centers, int64_t* chosen,
                               int cs, DeviceState* st, cudaStream_t s);
cudaError_t launch_lloyd(const float4* pts4, int64_t n, int k, int lloyd_iters, float4* centers, int32_t* labels,
                         double* sums, unsigned long long* changed, DeviceState* st, cudaStream_t s);
cudaError_t launch_label_stats(const float4* pts4, int64_t n, int k, const int32_t* labels, const float4* shift4,
                               double* stats64, DeviceState* st, cudaStream_t s);
cudaError_t launch_centers_out(const float4* centers4, int k, float* centers3, cudaStream_t s);

// ---------------------------------------------------------------- four dimensions (xyz + intensity)
// E-step parameters, pair-interleaved: components 2p, 2p+1 form pair p, which
// owns PAIR4_FLOATS floats at params[p * PAIR4_FLOATS] as float2 slots
// {comp 2p, comp 2p+1}:
//   slot 0..9   P' = alpha * L^{-1}, lower triangle (00,10,11,20,21,22,30,31,32,33)
//   slot 10     c = log2 w + sum_j log2 (L^{-1})_jj - (4/2) log2(2 pi)
//   slot 11..14 -mu (binary32; also the shift of the M-step statistics)
//   slot 15     w (N_b after an M-step, or the caller's weight)
//   slot 16     a lower bound of sigma_min(P')^2, as slot 14 in 3-D; slot 17 padding
// Statistics (NSTAT4, about y = P'(x - mu)): S0, S1[4], S2[10] in the order 00,01,02,03,11,12,13,22,23,33;
// binary64 model (MODEL4): w, mu[4], Sigma[10] in the same order.
constexpr int PAIR4_FLOATS = 36;
constexpr int SLOT4_P = 0, SLOT4_C = 10, SLOT4_NMU = 11, SLOT4_W = 15, SLOT4_S = 16;
constexpr int NSTAT4 = 15;
constexpr int MODEL4 = 15;
// index of (i, j), i <= j, in the upper-triangle order 00,01,02,03,11,12,13,22,23,33
__host__ __device__ constexpr int sym4(int i, int j) { return i * (7 - i) / 2 + j; }

// A 4-D fit's sums: whitened, with LOST_SUMS4 in DeviceState::error (no gira_status) where binary32 lost part
// of a covariance in them; about x - mu; whitened and not checked.
enum class Sums4 { Checked, About, Whitened };
constexpr int LOST_SUMS4 = -1;

// Component pairs the parameter buffer holds for k.
int params4_pairs(int k);
// N x 4 -> pts4 (x,y,z,I) (nullable) and pts8 (x,x,y,y)(z,z,I,I); flags non-finite input.
cudaError_t launch_pack4(const float* pts4in, int64_t n, float4* pts4, float4* pts8, DeviceState* st,
                         cudaStream_t s);
cudaError_t launch_fill_padding4(float* params, int k, cudaStream_t s);
// The dense E-step of little work (estep4_dense says for which n and k).
struct EStep4Launch {
    const float4* pts8;    // 2 float4 per point: (x,x,y,y) (z,z,I,I)
    int64_t n;
    int k;
    const float* params;
    int64_t pts_per_cta;   // multiple of 8
    float* partials;       // [grid][pairs][2 NSTAT4] (stats launches)
    double* ll_partials;   // [grid]
    float* per_point;      // [n] natural-log lse, or nullptr
    DeviceState* st;
    int iter;              // 1-based EM iteration; skipped when iter > st->stop_after
    bool world = false;    // statistics about x - mu, not whitened
};
bool estep4_dense(int64_t n, int k, bool stats);
int estep4_dense_grid(int64_t n, int k, int num_sms, int64_t* pts_per_cta);
cudaError_t launch_estep4_dense(const EStep4Launch& a, bool stats, int grid, cudaStream_t s, bool pdl = false);
// M-step from the partials of launch_reach_stats or launch_estep4_dense ([slices][pairs][2 NSTAT4],
// live where live2 says; nullptr: all) or, when partials is nullptr, from binary64 one-hot statistics stats64
// about shift4; sums as the partials are; em as in launch_reduce_finalize, the log-likelihood being the sum of
// llp[0 .. ll_count).  Slot b holds the caller's component perm[b] (nullptr: b).
cudaError_t launch_reduce_finalize4(const float* partials, const uint32_t* live2, int slices, const double* llp,
                                    int ll_count, const double* stats64, const float4* shift4, int k, int64_t n,
                                    double reg, double tol, double* model64, float* params, double* trace,
                                    const int* perm, DeviceState* st, int iter, bool em, cudaStream_t s,
                                    bool pdl = false, Sums4 sums = Sums4::Whitened);
// Components in Morton order of their means, as launch_order_components (scratch: k * MODEL4 doubles).
cudaError_t launch_order_components4(double* model64, double* scratch, int k, int* perm, float* params,
                                     DeviceState* st, cudaStream_t s);
// ctr, aux (nullable): as launch_model_points.
cudaError_t launch_params_from_model4(const float* w, const float* mu, const float* cov, int k, double* model64,
                                      float* params, float4* ctr, float2* aux, DeviceState* st, cudaStream_t s);
cudaError_t launch_model_out4(const double* model64, int k, float* w, float* mu, float* cov, const int* perm,
                              const DeviceState* st, cudaStream_t s);
// Lloyd in four dimensions and the one-hot statistics about the final centres.
cudaError_t launch_lloyd4(const float4* pts4, int64_t n, int k, int lloyd_iters, float4* centers, int32_t* labels,
                          double* sums, unsigned long long* changed, DeviceState* st, cudaStream_t s);
cudaError_t launch_label_stats4(const float4* pts4, int64_t n, int k, const int32_t* labels, const float4* shift4,
                                double* stats64, DeviceState* st, cudaStream_t s);
// Gaussian-mixture regression of the 4th coordinate on the first three.
int cond_floats();
bool conditional4_grouped(int64_t m, int k);   // whether it takes neighbours together (wants an order)
// order (nullable): the order in which the kernel takes the locations (any permutation gives
// the same results; one that keeps neighbours together is faster).
cudaError_t launch_conditional4(const float* locs, const int* order, int64_t m, int k, const float* w, const float* mu,
                                const float* cov, float* prep, float* cmean, float* cvar, DeviceState* st,
                                cudaStream_t s);
// m draws from a d-dimensional mixture (d = 3 or 4); cum: k doubles, chol: 16 k doubles.
cudaError_t launch_sample(int64_t m, int k, int d, const float* w, const float* mu, const float* cov, uint64_t seed,
                          double* cum, double* chol, float* out, int32_t* comp, DeviceState* st, cudaStream_t s);

// ---------------------------------------------------------------- mode seeking (K from a bandwidth)
// Temporary bytes the sorts / scans of one gira_gbms call need for n points.
size_t gbms_temp_bytes(int64_t n, int d);
// Points -> float4 copies, cell keys and identity indices; flags non-finite input
// (GIRA_ERR_NONFINITE_INPUT) and coordinates outside the cell range (GIRA_ERR_INVALID_ARG).
cudaError_t launch_gbms_keys(const float* pts, int64_t n, int d, double h, float4* pts4, uint64_t* keys, int* idx,
                             DeviceState* st, cudaStream_t s);
// Sort (key, index) pairs by key, then the distinct keys, their run lengths and
// starts; *ncells (device) receives the number of distinct keys.
cudaError_t gbms_sort_cells(void* temp, size_t temp_bytes, const uint64_t* keys_in, uint64_t* keys_out,
                            const int* idx_in, int* idx_out, int64_t n, int d, uint64_t* ukeys, int* ulen,
                            int* ustart, int* ncells, cudaStream_t s);
// Points in cell order.
cudaError_t launch_gbms_gather(const float4* pts4, const int* idx, int64_t n, float4* spts, cudaStream_t s);
// Hash table of the *ncells <= nmax cells (key, length << 32 | start): gbms_table_slots(nmax)
// slots.
unsigned gbms_table_slots(int64_t nmax);
cudaError_t launch_gbms_table(const uint64_t* ukeys, const int* ustart, const int* ulen, const int* ncells, int nmax,
                              ulonglong2* table, cudaStream_t s);
// The box of each cell's points at boxes[start], boxes[start + 1] (n entries; cells of one
// point have none).
cudaError_t launch_gbms_boxes(const float4* spts, const int* ustart, const int* ulen, int ncells, float4* boxes,
                              cudaStream_t s);
// One CTA per seed (cell): the seed's moves; modes[s] and counts[s] (0: dropped).  table: of
// nmax = ncells cells.
cudaError_t launch_gbms_shift(const float4* spts, const float4* boxes, const uint64_t* ukeys,
                              const ulonglong2* table, int64_t n, int ncells, int d, double h, int max_iter,
                              double4* modes, int* counts, const DeviceState* st, cudaStream_t s);
// Rank keys of the ns seeds (of n points) and their sort; *nlive (device, zeroed by the caller)
// receives the number of live modes.
cudaError_t launch_gbms_rank(void* temp, size_t temp_bytes, const int* counts, int64_t n, int ns, uint64_t* rkeys,
                             uint64_t* rkeys_sorted, int* nlive, cudaStream_t s);
// Live modes in rank order (rmodes, rcount), their cell keys and rank indices for
// the merge grid, and the merge state (undecided).
cudaError_t launch_gbms_rank_modes(const uint64_t* rkeys_sorted, const int* nlive, int nmax, const double4* modes,
                                   const int* counts, int d, double h, double4* rmodes, int* rcount, uint64_t* mkeys,
                                   int* midx, int* state, DeviceState* st, cudaStream_t s);
// One merge round; *undecided (zeroed by the caller) counts ranks still open.
cudaError_t launch_gbms_merge_round(const double4* rmodes, const int* nlive, int nmax, const ulonglong2* table,
                                    const int* midx_sorted, int d, double h, int* state, int* undecided,
                                    cudaStream_t s);
// Kept modes in rank order -> modes_out (k x d binary64) and counts_out (nullable);
// pos[r] is the output slot of rank r (exclusive sum of the kept flags).
cudaError_t launch_gbms_output(void* temp, size_t temp_bytes, const int* state, const int* nlive, int nmax,
                               const double4* rmodes, const int* rcount, int d, int* flags, int* pos,
                               double* modes_out, int* counts_out, cudaStream_t s);

// Test hook: one wait that nothing ends (mode 0: mbarrier, limit in ns; mode 1:
// global counter, limit in polls); counter and abort_flag: zeroed device ints.
cudaError_t launch_wait_probe(int mode, long long limit, int* counter, int* abort_flag, DeviceState* st,
                              cudaStream_t s);

// Set this thread's last-error message (msg may be nullptr to keep it) and
// component (what gira_last_error_message / gira_last_error_component return).
void record_error(const char* msg, int component);

// The status a call returns for the device status word it read back (GIRA_OK
// when no kernel recorded an error), with this thread's last-error message and,
// for GIRA_ERR_NOT_PD, the component.
gira_status device_status(const DeviceState& h);

// Name of the E-step kernel this host thread launched last (the runtime's name
// of the function, demangled; "" before the first launch).
const char* last_estep_kernel();
// Record fn (an E-step kernel about to be launched) as the last one.
void note_estep_kernel(const void* fn);

}  // namespace gira
