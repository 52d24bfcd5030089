// gbms_kernels.cu -- mode seeking that sets the number of components K.
//
// GIRA (arXiv 2307.00071) Sec. V, paragraph "Gaussian Blurring Mean Shift", and
// Fig. "information flow": seeds from a binned estimator, each seed moved to
// the average of the points within the bandwidth h of it until it stops moving
// (or an iteration limit), the distinct end points counted.  The paper queries
// neighbours with a kd-tree on the CPU; here the points are sorted by grid cell
// (cells of size h, the same cells that give the seeds) and a ball query looks the
// 3^D (at most 4^D) cells around the seed up in a hash table.
//
// Definitions taken by every step (both sides of the parity tests):
//   cell     c_i(x) = floor(x_i / h + 0.5) (binary64), |c_i| < 2^15;
//            key = sum_i (c_i + 2^15) 2^(16 i)
//   seeds    one per occupied cell, at c h, in ascending key order
//   ball     binary32 squared distance between x and (float)m in the order
//            ((d0^2 + d1^2) + d2^2) [+ d3^2], no FMA, <= (float)(h*h)
//   mean     exact 64-bit sums of rint(x_i 2^24) (|x_i| < 2^12), then
//            ((double)S / count) 2^-24: independent of the order of summation
//   stop     ||m_t - m_{t-1}||^2 <= (1e-3 h)^2 (binary64) or t = max_iter;
//            a seed whose ball is empty is dropped
//   merge    modes ranked by count (descending), ties by seed; in rank order a
//            mode is kept unless a kept mode lies within h (binary64 squared
//            distance, coordinate order, no FMA, <= h*h)
// The merge runs in rounds: a mode is kept once every earlier-ranked mode
// within h of it is known to be dropped, and dropped once one of them is kept;
// each round decides at least the lowest undecided rank, and the result is the
// sequential greedy one.
#include <float.h>
#include <limits.h>
#include <math.h>

#include <cub/cub.cuh>

#include "gira_internal.cuh"

namespace gira {

namespace {

constexpr unsigned FULL = 0xffffffffu;
constexpr int GB_WARPS = 8;          // warps (seeds or modes) per CTA
constexpr int GB_LOOKS = 16;         // looks of a merge round at the ranks it waits for
constexpr int GB_MAX_CELLS = 256;    // at most 4 cells per dimension, 4 dimensions
constexpr unsigned long long GB_EMPTY = ~0ull;
constexpr double Q_SCALE = 16777216.0;   // 2^24

__device__ __forceinline__ bool cell_of(double v, double h, int* c) {
    const double f = floor(__dadd_rn(__ddiv_rn(v, h), 0.5));
    if (!(f > -32768.0 && f < 32768.0)) return false;
    *c = (int)f;
    return true;
}

// cell_of for a binary32 v: where v / h + 0.5 in binary32 (within 4 2^-24 relative of v / h, and
// 2^-24 of the sum) is clearly between two integers, its floor is the binary64 one.
__device__ __forceinline__ bool cell_of_point(float v, double h, float inv_h, int* c) {
    const float q = v * inv_h, f = q + 0.5f, fl = floorf(f), frac = f - fl;
    const float err = fmaf(fabsf(q), 1e-6f, 1e-6f);
    if (fabsf(f) < 32000.f && frac > err && frac < 1.f - err) {
        *c = (int)fl;
        return true;
    }
    return cell_of((double)v, h, c);
}

__device__ __forceinline__ uint64_t key_of(const int* c, int d) {
    uint64_t k = 0;
    for (int i = 0; i < d; ++i) k |= (uint64_t)(uint32_t)(c[i] + 32768) << (16 * i);
    return k;
}

__device__ __forceinline__ int cell_coord(uint64_t key, int i) { return (int)((key >> (16 * i)) & 0xFFFFu) - 32768; }

// ---- the occupied cells as a hash table: slot (key, length << 32 | start), range GB_EMPTY where
// free, two slots per cell, linear probing.  A lookup is one or two dependent loads; a binary
// search of the sorted keys is fifteen (22,297 cells), and a seed that moves looks up to 256
// cells.
__device__ __forceinline__ unsigned gb_slot(uint64_t key, unsigned nslots) {
    key = (key ^ (key >> 32)) * 0x9E3779B97F4A7C15ull;   // the odd constant nearest 2^64 / golden ratio
    return (unsigned)__umul64hi((key ^ (key >> 29)) * 0x9E3779B97F4A7C15ull, nslots);
}

__global__ void gbms_table_kernel(const uint64_t* __restrict__ ukeys, const int* __restrict__ ustart,
                                  const int* __restrict__ ulen, const int* __restrict__ ncells, ulonglong2* table,
                                  unsigned nslots) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= *ncells) return;
    const uint64_t key = ukeys[i];
    const unsigned long long range = (unsigned long long)(unsigned)ulen[i] << 32 | (unsigned)ustart[i];
    unsigned at = gb_slot(key, nslots);
    for (unsigned probe = 0; probe < nslots; ++probe) {   // at most half the slots are taken
        if (atomicCAS(&table[at].y, GB_EMPTY, range) == GB_EMPTY) {
            table[at].x = key;
            return;
        }
        at = at + 1 < nslots ? at + 1 : 0;
    }
}

// the points of cell `key`: length << 32 | start, or 0 (no cell is empty); v, w: the slot at
// `at` and the next, loaded together
__device__ __forceinline__ unsigned long long gb_resolve(const ulonglong2* __restrict__ table, unsigned nslots,
                                                         uint64_t key, unsigned at, ulonglong2 v, ulonglong2 w) {
    for (unsigned probe = 0; probe < nslots; probe += 2) {
        if (v.y == GB_EMPTY) return 0ull;
        if (v.x == key) return v.y;
        if (w.y == GB_EMPTY) return 0ull;
        if (w.x == key) return w.y;
        at = at + 2 < nslots ? at + 2 : at + 2 - nslots;
        v = __ldg(table + at);
        w = __ldg(table + (at + 1 < nslots ? at + 1 : 0));
    }
    return 0ull;
}

// Sums of rint(x 2^24), |x| < 2^12, without a conversion (64-bit ones run at the binary64 rate,
// 32-bit ones at a quarter of the adders'): y = x 2^24 is exact in binary32; adding 1.5 2^38
// rounds it to a multiple of 2^15, hi, whose integer hi / 2^15 is the difference of the sum's
// bits and the constant's; lo = y - hi is exact (|lo| <= 2^14), and adding 1.5 2^23 rounds it to
// an integer the same way, ties to even as those of y (hi and both constants are even).  The
// constants' bits are taken off, count times, when the 32-bit sums are added to 64-bit ones:
// |hi / 2^15| < 2^21 and so after at most 512 points.
struct GbSum {
    static constexpr float HI = 412316860416.f, LO = 12582912.f;   // 1.5 2^38, 1.5 2^23
    int cnt = 0;
    unsigned hi[4] = {0u, 0u, 0u, 0u}, lo[4] = {0u, 0u, 0u, 0u};
    __device__ __forceinline__ void add1(float x, int i) {
        const float t = __fmaf_rn(x, 16777216.f, HI);
        hi[i] += __float_as_uint(t);
        lo[i] += __float_as_uint(__fadd_rn(__fmaf_rn(x, 16777216.f, -__fsub_rn(t, HI)), LO));
    }
    __device__ __forceinline__ void add(float4 x, int d) {
        ++cnt;
        add1(x.x, 0);
        add1(x.y, 1);
        add1(x.z, 2);
        if (d == 4) add1(x.w, 3);
    }
    __device__ __forceinline__ void flush(int& total, long long (&sum)[4], int d) {
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const unsigned c = i < d ? (unsigned)cnt : 0u;
            sum[i] += ((long long)(int)(hi[i] - c * __float_as_uint(HI)) << 15) +
                      (int)(lo[i] - c * __float_as_uint(LO));
            hi[i] = lo[i] = 0u;
        }
        total += cnt;
        cnt = 0;
    }
};

__device__ __forceinline__ float dist2_ball(float4 x, const float* mf, int d) {
    const float d0 = __fsub_rn(x.x, mf[0]), d1 = __fsub_rn(x.y, mf[1]), d2 = __fsub_rn(x.z, mf[2]);
    float s = __fadd_rn(__fadd_rn(__fmul_rn(d0, d0), __fmul_rn(d1, d1)), __fmul_rn(d2, d2));
    if (d == 4) {
        const float d3 = __fsub_rn(x.w, mf[3]);
        s = __fadd_rn(s, __fmul_rn(d3, d3));
    }
    return s;
}

__device__ __forceinline__ double dist2_modes(const double* a, const double* b, int d) {
    double s = 0.0;
    for (int i = 0; i < d; ++i) {
        const double dv = __dsub_rn(a[i], b[i]);
        s = (i == 0) ? __dmul_rn(dv, dv) : __dadd_rn(s, __dmul_rn(dv, dv));
    }
    return s;
}

// The cells a ball of radius h around m can touch: per dimension [lo_i, lo_i + nr_i).
// Only a superset is needed (the ball test decides membership), so binary32
// with the radius inflated by 5 % suffices: the binary32 error of m_i / h is
// below 4e-3 cells for every |c_i| < 2^15, far inside the margin, and a point
// in the ball lies within h (1 + 2^-23) of m in every coordinate.  r: the radius, at most
// 1.35 h (then 2.1 r / h < 3 and there are at most four cells per dimension).
__device__ __forceinline__ int ball_cells(const float* m, int d, float r, float inv_h, int* lo, int* nr) {
    const float hin = 1.05f * r;
    int total = 1;
    for (int i = 0; i < d; ++i) {
        const float a = floorf(fmaf(m[i] - hin, inv_h, 0.5f));
        const float b = floorf(fmaf(m[i] + hin, inv_h, 0.5f));
        const int la = (int)fmaxf(a, -32767.f), lb = (int)fminf(b, 32767.f);
        lo[i] = la;
        nr[i] = lb >= la ? lb - la + 1 : 0;
        total *= nr[i];
    }
    return total;
}

// key of candidate t of the box [lo, lo + nr)
__device__ __forceinline__ uint64_t gb_candidate(const int* lo, const int* nr, int d, int t) {
    int c[4] = {0, 0, 0, 0};
    for (int i = 0; i < d; ++i) {
        c[i] = lo[i] + t % nr[i];
        t /= nr[i];
    }
    return key_of(c, d);
}

// Lanes list the occupied cells of the candidate box (start, length) in the
// warp's shared arrays and fill pre[] with the exclusive prefix of the lengths
// (pre[count] = total points); returns the count.
__device__ int gather_cells(const ulonglong2* __restrict__ table, unsigned nslots, const int* lo, const int* nr,
                            int total, int d, int lane, int* cs, int* pre) {
    int nfound = 0;
    for (int base = 0; base < total; base += 128) {
        uint64_t key[4];
        unsigned at[4];
        ulonglong2 v[4], w[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) {   // the first probes together
            const int t = base + 32 * u + lane;
            v[u].y = GB_EMPTY;
            if (t < total) {
                key[u] = gb_candidate(lo, nr, d, t);
                at[u] = gb_slot(key[u], nslots);
                v[u] = __ldg(table + at[u]);
                w[u] = __ldg(table + (at[u] + 1 < nslots ? at[u] + 1 : 0));
            }
        }
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            const unsigned long long range =
                v[u].y == GB_EMPTY ? 0ull : gb_resolve(table, nslots, key[u], at[u], v[u], w[u]);
            const unsigned mk = __ballot_sync(FULL, range != 0ull);
            if (range) {
                const int f = nfound + __popc(mk & ((1u << lane) - 1u));
                cs[f] = (int)(unsigned)range;
                pre[f] = (int)(range >> 32);   // lengths for now
            }
            nfound += __popc(mk);
        }
    }
    __syncwarp();
    // exclusive prefix of the lengths, 32 at a time
    int carry = 0;
    for (int base = 0; base < nfound; base += 32) {
        const int j = base + lane;
        const int v = (j < nfound) ? pre[j] : 0;
        int inc = v;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int u = __shfl_up_sync(FULL, inc, o);
            if (lane >= o) inc += u;
        }
        __syncwarp();
        if (j < nfound) pre[j] = carry + inc - v;
        carry += __shfl_sync(FULL, inc, 31);
    }
    if (lane == 0) pre[nfound] = carry;
    __syncwarp();
    return nfound;
}

// index j with pre[j] <= t < pre[j + 1]
__device__ __forceinline__ int cell_of_flat(const int* pre, int n, int t) {
    int lo = 0, hi = n - 1;
    while (lo < hi) {
        const int mid = (lo + hi + 1) >> 1;
        if (pre[mid] <= t) lo = mid; else hi = mid - 1;
    }
    return lo;
}

__global__ void gbms_keys_kernel(const float* __restrict__ pts, int64_t n, int d, double h, float4* pts4,
                                 uint64_t* keys, int* idx, DeviceState* st) {
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    float v[4] = {0.f, 0.f, 0.f, 0.f};
    int c[4] = {0, 0, 0, 0};
    bool ok = true, fin = true;
    const float inv_h = 1.0f / (float)h;
    for (int j = 0; j < d; ++j) {
        v[j] = pts[(size_t)d * i + j];
        fin = fin && isfinite(v[j]);
        ok = ok && fabsf(v[j]) < 4096.0f && cell_of_point(v[j], h, inv_h, &c[j]);
    }
    if (!fin) set_error(st, GIRA_ERR_NONFINITE_INPUT);
    else if (!ok) set_error(st, GIRA_ERR_INVALID_ARG);
    pts4[i] = make_float4(v[0], v[1], v[2], v[3]);
    keys[i] = key_of(c, d);
    idx[i] = (int)i;
}

// Points in cell order.
__global__ void gbms_gather_kernel(const float4* __restrict__ pts4, const int* __restrict__ idx, int64_t n,
                                   float4* spts) {
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) spts[i] = pts4[idx[i]];
}

// The box of each cell's points, where the cell has more than one: boxes[start] and
// boxes[start + 1] of its points' places (a warp per cell).
__global__ void gbms_box_kernel(const float4* __restrict__ spts, const int* __restrict__ ustart,
                                const int* __restrict__ ulen, int ncells, float4* boxes) {
    const int i = (int)((blockIdx.x * blockDim.x + threadIdx.x) >> 5), lane = threadIdx.x & 31;
    if (i >= ncells) return;
    const int start = ustart[i], len = ulen[i];
    if (len < 2) return;
    float4 lo = spts[start], hi = lo;
    for (int q = lane; q < len; q += 32) {
        const float4 x = spts[start + q];
        lo = make_float4(fminf(lo.x, x.x), fminf(lo.y, x.y), fminf(lo.z, x.z), fminf(lo.w, x.w));
        hi = make_float4(fmaxf(hi.x, x.x), fmaxf(hi.y, x.y), fmaxf(hi.z, x.z), fmaxf(hi.w, x.w));
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        lo.x = fminf(lo.x, __shfl_xor_sync(FULL, lo.x, o));
        lo.y = fminf(lo.y, __shfl_xor_sync(FULL, lo.y, o));
        lo.z = fminf(lo.z, __shfl_xor_sync(FULL, lo.z, o));
        lo.w = fminf(lo.w, __shfl_xor_sync(FULL, lo.w, o));
        hi.x = fmaxf(hi.x, __shfl_xor_sync(FULL, hi.x, o));
        hi.y = fmaxf(hi.y, __shfl_xor_sync(FULL, hi.y, o));
        hi.z = fmaxf(hi.z, __shfl_xor_sync(FULL, hi.z, o));
        hi.w = fmaxf(hi.w, __shfl_xor_sync(FULL, hi.w, o));
    }
    if (lane == 0) {
        boxes[start] = lo;
        boxes[start + 1] = hi;
    }
}

// One CTA of T threads per seed: the moves of the seed of cell ukeys[s] (see the header).
// What bounds it is the latency of a move, moves being serial.  Most seeds have little work
// (12 moves, 680 candidate points and 200 in the ball on average for a 4-D frame at h = 0.05);
// a few hundred in dense flat parts move up to max_iter times among thousands of points.
//  - The threads look the candidate cells up in the hash table at once, and the cells are
//    kept while the seed stays among them.
//  - Up to CAP candidate points are copied into shared memory (cp.async, all in flight
//    together) and swept there by this and the following moves.
//  - More than CAP are swept in global memory, with an anchor: points
//    within h - rho of the seed's place a stay in the ball, and those beyond h + rho out of
//    it, while the seed is within rho of a.  The first are summed once (each thread keeps its
//    part), the shell between goes to shared memory, and only that is swept until the seed
//    leaves.  rho is 24 of the seed's last step, at most what the shell's room and the
//    cells allow.
//  - 64-bit sums over a warp are three 32-bit warp reductions of 24-bit parts.
//  - Binary64 work (the move and its stopping test) is one warp's, lane i for coordinate i:
//    GB300 runs binary64 at a small fraction of binary32.
// Any order of the points gives the same exact sums.  Measured: 276,348 points of a 4-D frame,
// h = 0.05, 22,297 seeds: 9.7 to 11 ms when warp 0 searched the sorted keys and every move read
// every candidate from global memory through a walk over the cells' prefix; 1 to 5 ms now,
// by the scene (starting the seeds of dense cells first did not shorten the tail).
constexpr int GB_CELL_LANES = 8;   // lanes that copy one cell
constexpr float GB_STEPS = 24.f;   // rho in last steps: a sweep for an anchor costs some 30 of its shell
constexpr float GB_MARGIN = 1e-5f;   // relative, against the binary32 rounding of distances (5e-7)

constexpr int GB_CHUNKS = 1024;      // pieces of cells a sweep of global memory is cut into

template <int T, int CAP>
__global__ void __launch_bounds__(T) gbms_shift_kernel(const float4* __restrict__ spts,
                                                       const float4* __restrict__ boxes,
                                                       const uint64_t* __restrict__ ukeys,
                                                       const ulonglong2* __restrict__ table, unsigned nslots, int d,
                                                       double h, int max_iter, double4* modes, int* counts,
                                                       const DeviceState* st) {
    constexpr int W = T / 32;
    extern __shared__ __align__(16) float4 s_pts[];   // CAP
    __shared__ int s_cs[GB_MAX_CELLS], s_len[GB_MAX_CELLS], s_off[GB_MAX_CELLS];
    __shared__ unsigned long long s_cells;   // cells << 32 | points
    __shared__ int2 s_chunk[GB_CHUNKS];      // start, length
    __shared__ int s_nshell, s_nchunk;
    __shared__ long long s_red[W][5];
    __shared__ double s_m[4];
    __shared__ float s_mf[4];
    __shared__ float s_rho;   // of the next (or present) anchor, 0: none
    __shared__ int s_lo[4], s_nr[4];
    __shared__ int s_moved;    // the candidate cells are to be looked up
    __shared__ int s_shell;    // the shell in shared memory holds for the seed's place
    __shared__ int s_done, s_count;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int s = blockIdx.x;
    if (st->error) return;   // set before the launch: uniform
    const float hf = (float)h, inv_hf = 1.0f / hf;
    const float h2f = __double2float_rn(__dmul_rn(h, h));
    // warp 0: the cells of the ball of radius r around the seed (lane i has coordinate i)
    auto place_cells = [&](float mf, float r) {
        int lo = INT_MIN, nr = 0;
        if (lane < d) ball_cells(&mf, 1, r, inv_hf, &lo, &nr);
        const bool any = __any_sync(FULL, lane < d && (lo != s_lo[lane] || nr != s_nr[lane]));
        if (lane < d) {
            s_lo[lane] = lo;
            s_nr[lane] = nr;
        }
        if (lane == 0) {
            s_moved = any;
            if (any) s_cells = 0ull;
        }
    };
    if (warp == 0) {
        const uint64_t key = ukeys[s];
        if (lane < 4) {
            const double m0 = lane < d ? __dmul_rn((double)cell_coord(key, lane), h) : 0.0;
            s_m[lane] = m0;
            s_mf[lane] = __double2float_rn(m0);
            s_lo[lane] = INT_MIN;
            s_nr[lane] = 0;
        }
        if (lane == 0) {
            s_done = s_count = s_shell = s_nshell = s_nchunk = 0;
            s_rho = 0.f;
        }
        __syncwarp();
        place_cells(lane < 4 ? s_mf[lane] : 0.f, hf);
    }
    const double thr = __dmul_rn(1e-3, h), thr2 = __dmul_rn(thr, thr);
    int base_cnt = 0;   // this thread's part of the points that stay in the ball
    long long base_sum[4] = {0, 0, 0, 0};
    float a = 0.f;      // warp 0, lane i: coordinate i of the anchor
    __syncthreads();
    for (int t = 1; t <= max_iter; ++t) {
        if (s_moved) {   // uniform
            int lo[4], nr[4], total = 1;
            for (int i = 0; i < d; ++i) {
                lo[i] = s_lo[i];
                nr[i] = s_nr[i];
                total *= nr[i];
            }
            for (int q0 = 32 * warp; q0 < total; q0 += T) {
                unsigned long long range = 0ull;
                if (q0 + lane < total) {
                    const uint64_t key = gb_candidate(lo, nr, d, q0 + lane);
                    const unsigned at = gb_slot(key, nslots);
                    range = gb_resolve(table, nslots, key, at, __ldg(table + at),
                                       __ldg(table + (at + 1 < nslots ? at + 1 : 0)));
                }
                const int len = (int)(range >> 32);
                const unsigned mk = __ballot_sync(FULL, len > 0);
                if (!mk) continue;
                int inc = len;   // inclusive sum over the lanes
#pragma unroll
                for (int o = 1; o < 32; o <<= 1) {
                    const int u = __shfl_up_sync(FULL, inc, o);
                    if (lane >= o) inc += u;
                }
                unsigned long long both = 0ull;
                if (lane == 31) both = atomicAdd(&s_cells, (unsigned long long)__popc(mk) << 32 | (unsigned)inc);
                both = __shfl_sync(FULL, both, 31);
                const int at = (int)(both >> 32) + __popc(mk & ((1u << lane) - 1u));
                const int off = (int)(unsigned)both + inc - len;
                if (len > 0) {
                    s_cs[at] = (int)(unsigned)range;
                    s_len[at] = len;
                    s_off[at] = off;
                }
            }
            __syncthreads();
            if ((int)(unsigned)s_cells <= CAP) {
                const int nf = (int)(s_cells >> 32);
                for (int j = tid / GB_CELL_LANES; j < nf; j += T / GB_CELL_LANES) {
                    const int len = s_len[j];
                    const float4* src = spts + s_cs[j];
                    const unsigned dst = (unsigned)__cvta_generic_to_shared(s_pts + s_off[j]);
                    for (int q = tid % GB_CELL_LANES; q < len; q += GB_CELL_LANES)
                        asm volatile("cp.async.ca.shared.global [%0], [%1], 16;" ::"r"(dst + 16u * q), "l"(src + q)
                                     : "memory");
                }
                asm volatile("cp.async.wait_all;" ::: "memory");
                __syncthreads();
            }
        }
        const float mf[4] = {s_mf[0], s_mf[1], s_mf[2], s_mf[3]};
        const int npts = (int)(unsigned)s_cells;
        int cnt = 0;
        long long sum[4] = {0, 0, 0, 0};
        GbSum acc;
        // each(x, valid) for the candidates in global memory, but for cells whose box is farther than
        // reach2 (rounding is monotone: no point of such a cell is computed nearer).  The cells are
        // cut into chunks of a multiple of 32 points; a warp takes four chunks at a time.
        auto sweep_global = [&](float reach2, int& total, long long (&into)[4], auto&& each) {
            const int nf = (int)(s_cells >> 32);
            const int size = 32 * ((npts + 32 * (GB_CHUNKS - GB_MAX_CELLS) - 1) / (32 * (GB_CHUNKS - GB_MAX_CELLS)));
            for (int j = tid; j < nf; j += T) {
                const int start = s_cs[j], len = s_len[j];
                float4 lo, hi;
                if (len > 1) {
                    lo = __ldg(boxes + start);
                    hi = __ldg(boxes + start + 1);
                } else {
                    lo = hi = __ldg(spts + start);
                }
                const float4 near = make_float4(fminf(fmaxf(mf[0], lo.x), hi.x), fminf(fmaxf(mf[1], lo.y), hi.y),
                                                fminf(fmaxf(mf[2], lo.z), hi.z), fminf(fmaxf(mf[3], lo.w), hi.w));
                if (dist2_ball(near, mf, d) > reach2) continue;
                const int nch = (len + size - 1) / size, at = atomicAdd(&s_nchunk, nch);   // <= GB_CHUNKS in all
                for (int c = 0; c < nch; ++c) s_chunk[at + c] = make_int2(start + c * size, min(size, len - c * size));
            }
            __syncthreads();
            const int nchunk = s_nchunk;
            int trips = 0;
            for (int c0 = 4 * warp; c0 < nchunk; c0 += 4 * W) {
                int2 ch[4];
#pragma unroll
                for (int u = 0; u < 4; ++u) ch[u] = c0 + u < nchunk ? s_chunk[c0 + u] : make_int2(s_chunk[c0].x, 0);
                for (int q = lane; q - lane < size; q += 32) {
                    float4 x[4];
                    bool valid[4];
#pragma unroll
                    for (int u = 0; u < 4; ++u) {
                        valid[u] = q < ch[u].y;
                        x[u] = spts[ch[u].x + (valid[u] ? q : 0)];
                    }
                    each(x, valid);
                    if ((++trips & 63) == 0) acc.flush(total, into, d);
                }
            }
            acc.flush(total, into, d);
        };
        int swept = npts;   // points in shared memory to sweep
        if (npts > CAP) {
            bool shell = s_shell != 0;   // uniform
            const float rho = s_rho;
            if (!shell && rho > 0.f) {   // a new anchor
                const float in = (hf - rho) * (1.f - GB_MARGIN), out = (hf + rho) * (1.f + GB_MARGIN);
                const float in2 = in * in, out2 = out * out;
                base_cnt = 0;
                base_sum[0] = base_sum[1] = base_sum[2] = base_sum[3] = 0;
                sweep_global(out2, base_cnt, base_sum, [&](const float4 (&x)[4], const bool (&valid)[4]) {
                    unsigned mk[4];
                    int n = 0;
#pragma unroll
                    for (int u = 0; u < 4; ++u) {
                        const float q = dist2_ball(x[u], mf, d);
                        if (valid[u] && q <= in2) acc.add(x[u], d);
                        mk[u] = __ballot_sync(FULL, valid[u] && q > in2 && q <= out2);
                        n += __popc(mk[u]);
                    }
                    if (n == 0) return;
                    int at = 0;
                    if (lane == 0) at = atomicAdd(&s_nshell, n);
                    at = __shfl_sync(FULL, at, 0);
#pragma unroll
                    for (int u = 0; u < 4; ++u) {
                        const int w = at + __popc(mk[u] & ((1u << lane) - 1u));
                        if ((mk[u] >> lane & 1u) && w < CAP) s_pts[w] = x[u];
                        at += __popc(mk[u]);
                    }
                });
                if (lane < 4) a = s_mf[lane];
                __syncthreads();
                shell = s_nshell <= CAP;
            }
            if (shell) {
                cnt = base_cnt;
#pragma unroll
                for (int i = 0; i < 4; ++i) sum[i] = base_sum[i];
                swept = s_nshell;
            } else {
                swept = 0;
                if (rho > 0.f) {   // there was no room for the shell
                    if (tid == 0) s_nchunk = 0;
                    __syncthreads();
                }
                sweep_global(h2f, cnt, sum, [&](const float4 (&x)[4], const bool (&valid)[4]) {
#pragma unroll
                    for (int u = 0; u < 4; ++u)
                        if (valid[u] && dist2_ball(x[u], mf, d) <= h2f) acc.add(x[u], d);
                });
            }
        }
#pragma unroll 4
        for (int f = tid; f < swept; f += T) {
            const float4 x = s_pts[f];
            if (dist2_ball(x, mf, d) <= h2f) acc.add(x, d);   // CAP / T of them at most
        }
        acc.flush(cnt, sum, d);
        cnt = (int)__reduce_add_sync(FULL, (unsigned)cnt);
        if (lane == 0) s_red[warp][0] = cnt;
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const unsigned long long v = (unsigned long long)sum[i];
            const unsigned p0 = __reduce_add_sync(FULL, (unsigned)v & 0xFFFFFFu);
            const unsigned p1 = __reduce_add_sync(FULL, (unsigned)(v >> 24) & 0xFFFFFFu);
            const unsigned p2 = __reduce_add_sync(FULL, (unsigned)(v >> 48));   // modulo 2^16 suffices
            if (lane == 0)
                s_red[warp][1 + i] = (long long)((unsigned long long)p0 + ((unsigned long long)p1 << 24) +
                                                 ((unsigned long long)p2 << 48));
        }
        __syncthreads();
        if (warp == 0) {
            // the move: lane i < d takes coordinate i (one binary64 instruction serves
            // every coordinate), lane 0 sums the squared steps in coordinate order
            long long tot = 0;
            if (lane < 5)
                for (int w = 0; w < W; ++w) tot += s_red[w][lane];
            const long long count = __shfl_sync(FULL, tot, 0);
            const long long si = __shfl_down_sync(FULL, tot, 1);   // lane i: sum of coordinate i
            if (count == 0) {
                if (lane == 0) {
                    s_count = 0;
                    s_done = 1;
                }
            } else {
                double sq = 0.0, v = 0.0;
                if (lane < d) {
                    v = __dmul_rn(__ddiv_rn(__ll2double_rn(si), (double)count), 1.0 / Q_SCALE);
                    const double dv = __dsub_rn(v, s_m[lane]);
                    sq = __dmul_rn(dv, dv);
                }
                const double sq1 = __shfl_sync(FULL, sq, 1), sq2 = __shfl_sync(FULL, sq, 2),
                             sq3 = __shfl_sync(FULL, sq, 3);
                const float vf = __double2float_rn(v);
                __syncwarp();
                if (lane < d) {
                    s_m[lane] = v;
                    s_mf[lane] = vf;
                }
                float step2 = -1.f;   // of the move; negative: the last one
                if (lane == 0) {
                    double mv = __dadd_rn(__dadd_rn(sq, sq1), sq2);
                    if (d == 4) mv = __dadd_rn(mv, sq3);
                    s_count = (int)count;
                    if (mv <= thr2 || t == max_iter) s_done = 1;
                    else step2 = fmaxf(0.f, __double2float_rn(mv));
                }
                step2 = __shfl_sync(FULL, step2, 0);
                if (step2 >= 0.f) {
                    const bool large = npts > CAP;
                    const int nshell = s_nshell;
                    const float rho = s_rho;
                    float away = lane < d ? (vf - a) * (vf - a) : 0.f;   // |seed - anchor|^2
                    away += __shfl_xor_sync(FULL, away, 1);
                    away += __shfl_xor_sync(FULL, away, 2);
                    away = __shfl_sync(FULL, away, 0);
                    const float r = rho * (1.f - GB_MARGIN);
                    const bool hold = large && rho > 0.f && nshell <= CAP && away <= r * r;
                    __syncwarp();
                    if (hold) {
                        if (lane == 0) {
                            s_shell = 1;
                            s_moved = 0;
                        }
                    } else {
                        // the room: a shell of a flat part holds 4 rho / h of the ball's points;
                        // nothing below where squares lose bits
                        float next = 0.f;
                        if (large && h2f > 1e-30f)
                            next = fminf(fminf(GB_STEPS * sqrtf(step2), 0.35f * hf),
                                         hf * ((float)CAP / 4.5f) / (float)count);
                        if (nshell > CAP) next = fminf(next, 0.5f * rho);   // there was no room
                        if (next * next < 4.f * step2) next = 0.f;          // would not hold for two moves
                        if (lane == 0) {
                            s_shell = 0;
                            s_nshell = s_nchunk = 0;
                            s_rho = next;
                        }
                        place_cells(vf, hf + next);
                    }
                }
            }
        }
        __syncthreads();
        if (s_done) break;
    }
    if (tid == 0) {
        modes[s] = make_double4(s_m[0], s_m[1], s_m[2], s_m[3]);
        counts[s] = s_count;
    }
}

// Rank keys: (2^31 - 1 - count, seed) for live modes; dropped seeds sort last.
__global__ void gbms_rank_keys_kernel(const int* __restrict__ counts, int ns, uint64_t* rkeys, int* nlive) {
    const int s = blockIdx.x * blockDim.x + threadIdx.x;
    if (s >= ns) return;
    const int c = counts[s];
    rkeys[s] = c > 0 ? ((uint64_t)(0x7FFFFFFF - c) << 32) | (uint32_t)s : ~0ull;
    if (c > 0) atomicAdd(nlive, 1);
}

// Rank r: its mode, count and cell key (for the merge grid).
__global__ void gbms_rank_modes_kernel(const uint64_t* __restrict__ rkeys_sorted, const int* __restrict__ nlive,
                                       const double4* __restrict__ modes, const int* __restrict__ counts, int d,
                                       double h, double4* rmodes, int* rcount, uint64_t* mkeys, int* midx,
                                       int* state, DeviceState* st) {
    const int r = blockIdx.x * blockDim.x + threadIdx.x;
    if (r >= *nlive) return;
    const int s = (int)(rkeys_sorted[r] & 0xFFFFFFFFull);
    const double4 m = modes[s];
    rmodes[r] = m;
    rcount[r] = counts[s];
    const double mv[4] = {m.x, m.y, m.z, m.w};
    int c[4] = {0, 0, 0, 0};
    bool ok = true;
    for (int i = 0; i < d; ++i) ok = ok && cell_of(mv[i], h, &c[i]);
    if (!ok) set_error(st, GIRA_ERR_INVALID_ARG);   // unreachable: a mean of points lies inside their cells
    mkeys[r] = key_of(c, d);
    midx[r] = r;
    state[r] = 0;
}

// One merge round over the undecided ranks (state 0 undecided, 1 kept, 2 dropped), a warp each.
// Bound by the chain of ranks that wait for one another; looking again within a launch took
// the 22,297 modes of a frame from 17 launches of 20 us to two of 66.
__global__ void __launch_bounds__(GB_WARPS * 32) gbms_merge_round_kernel(
    const double4* __restrict__ rmodes, const int* __restrict__ nlive, const ulonglong2* __restrict__ table,
    unsigned nslots, const int* __restrict__ midx_sorted, int d, double h, int* state, int* undecided) {
    __shared__ int s_cs[GB_WARPS][GB_MAX_CELLS];
    __shared__ int s_pre[GB_WARPS][GB_MAX_CELLS + 1];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int r = blockIdx.x * GB_WARPS + warp;
    if (r >= *nlive) return;
    volatile int* vstate = state;
    if (vstate[r] != 0) return;   // warp-uniform read of a decided rank
    const double4 mr = rmodes[r];
    const double a[4] = {mr.x, mr.y, mr.z, mr.w};
    const double h2 = __dmul_rn(h, h);
    const float af[4] = {(float)mr.x, (float)mr.y, (float)mr.z, (float)mr.w};
    int lo[4], nr[4];
    const int total = ball_cells(af, d, (float)h, 1.0f / (float)h, lo, nr);
    const int nf = gather_cells(table, nslots, lo, nr, total, d, lane, s_cs[warp], s_pre[warp]);
    const int nmodes = s_pre[warp][nf];
    // The ranks it depends on are lower, so their warps were started before this one: it looks again
    // a few times (no more: they may be waiting as well) before it leaves the rank to the next
    // launch.  Within a cell the ranks rise.
    bool kept_near = false, pending = false;
    for (int look = 0; look < GB_LOOKS; ++look) {
        kept_near = pending = false;
        for (int f0 = 0; f0 < nmodes && !kept_near; f0 += 32) {
            const int f = f0 + lane;
            int so = 2;
            if (f < nmodes) {
                const int j = cell_of_flat(s_pre[warp], nf, f);
                const int o = midx_sorted[s_cs[warp][j] + (f - s_pre[warp][j])];
                if (o < r) {
                    const double4 mo = rmodes[o];
                    const double b[4] = {mo.x, mo.y, mo.z, mo.w};
                    so = vstate[o];
                    if (so != 2 && !(dist2_modes(a, b, d) <= h2)) so = 2;
                }
            }
            kept_near = __any_sync(FULL, so == 1);
            pending = pending || __any_sync(FULL, so == 0);
        }
        if (kept_near || !pending) break;
    }
    if (lane == 0) {
        if (kept_near) {
            vstate[r] = 2;
        } else if (!pending) {
            vstate[r] = 1;
        } else {
            atomicAdd(undecided, 1);
        }
    }
}

__global__ void gbms_kept_flags_kernel(const int* __restrict__ state, const int* __restrict__ nlive, int nmax,
                                       int* flags) {
    const int r = blockIdx.x * blockDim.x + threadIdx.x;
    if (r < nmax) flags[r] = (r < *nlive && state[r] == 1) ? 1 : 0;
}

__global__ void gbms_output_kernel(const int* __restrict__ flags, const int* __restrict__ pos,
                                   const int* __restrict__ nlive, const double4* __restrict__ rmodes,
                                   const int* __restrict__ rcount, int d, double* modes_out, int* counts_out) {
    const int r = blockIdx.x * blockDim.x + threadIdx.x;
    if (r >= *nlive || !flags[r]) return;
    const int k = pos[r];
    const double4 m = rmodes[r];
    const double mv[4] = {m.x, m.y, m.z, m.w};
    if (modes_out)
        for (int i = 0; i < d; ++i) modes_out[(size_t)d * k + i] = mv[i];
    if (counts_out) counts_out[k] = rcount[r];
}

}  // namespace

// ------------------------------------------------------------------ host side
size_t gbms_temp_bytes(int64_t n, int d) {
    size_t a = 0, b = 0, c = 0, e = 0;
    const int nn = (int)n;
    cub::DeviceRadixSort::SortPairs(nullptr, a, (const uint64_t*)nullptr, (uint64_t*)nullptr, (const int*)nullptr,
                                    (int*)nullptr, nn, 0, 16 * d);
    cub::DeviceRunLengthEncode::Encode(nullptr, b, (const uint64_t*)nullptr, (uint64_t*)nullptr, (int*)nullptr,
                                       (int*)nullptr, nn);
    cub::DeviceScan::ExclusiveSum(nullptr, c, (const int*)nullptr, (int*)nullptr, nn);
    cub::DeviceRadixSort::SortKeys(nullptr, e, (const uint64_t*)nullptr, (uint64_t*)nullptr, nn);
    return std::max(std::max(a, b), std::max(c, e));
}

cudaError_t launch_gbms_keys(const float* pts, int64_t n, int d, double h, float4* pts4, uint64_t* keys, int* idx,
                             DeviceState* st, cudaStream_t s) {
    gbms_keys_kernel<<<(unsigned)((n + 255) / 256), 256, 0, s>>>(pts, n, d, h, pts4, keys, idx, st);
    return cudaGetLastError();
}

cudaError_t gbms_sort_cells(void* temp, size_t temp_bytes, const uint64_t* keys_in, uint64_t* keys_out,
                            const int* idx_in, int* idx_out, int64_t n, int d, uint64_t* ukeys, int* ulen,
                            int* ustart, int* ncells, cudaStream_t s) {
    size_t tb = temp_bytes;
    cudaError_t e = cub::DeviceRadixSort::SortPairs(temp, tb, keys_in, keys_out, idx_in, idx_out, (int)n, 0, 16 * d, s);
    if (e != cudaSuccess) return e;
    tb = temp_bytes;
    e = cub::DeviceRunLengthEncode::Encode(temp, tb, keys_out, ukeys, ulen, ncells, (int)n, s);
    if (e != cudaSuccess) return e;
    tb = temp_bytes;
    return cub::DeviceScan::ExclusiveSum(temp, tb, ulen, ustart, (int)n, s);
}

cudaError_t launch_gbms_gather(const float4* pts4, const int* idx, int64_t n, float4* spts, cudaStream_t s) {
    gbms_gather_kernel<<<(unsigned)((n + 255) / 256), 256, 0, s>>>(pts4, idx, n, spts);
    return cudaGetLastError();
}

unsigned gbms_table_slots(int64_t nmax) { return (unsigned)(2 * nmax); }   // nmax <= 2^30

cudaError_t launch_gbms_table(const uint64_t* ukeys, const int* ustart, const int* ulen, const int* ncells, int nmax,
                              ulonglong2* table, cudaStream_t s) {
    const unsigned nslots = gbms_table_slots(nmax);
    const cudaError_t e = cudaMemsetAsync(table, 0xff, sizeof(ulonglong2) * (size_t)nslots, s);
    if (e != cudaSuccess) return e;
    gbms_table_kernel<<<(nmax + 255) / 256, 256, 0, s>>>(ukeys, ustart, ulen, ncells, table, nslots);
    return cudaGetLastError();
}

cudaError_t launch_gbms_boxes(const float4* spts, const int* ustart, const int* ulen, int ncells, float4* boxes,
                              cudaStream_t s) {
    gbms_box_kernel<<<(ncells + 7) / 8, 256, 0, s>>>(spts, ustart, ulen, ncells, boxes);
    return cudaGetLastError();
}

cudaError_t launch_gbms_shift(const float4* spts, const float4* boxes, const uint64_t* ukeys,
                              const ulonglong2* table, int64_t n, int ncells, int d, double h, int max_iter,
                              double4* modes, int* counts, const DeviceState* st, cudaStream_t s) {
    const unsigned nslots = gbms_table_slots(ncells);
    // a seed sees some ten cells' points (3 by 3 of a surface, and its neighbours): up to 64
    // points per cell 128 threads have a few each; above, there are fewer seeds with longer sweeps
    constexpr int CAP = 2048;   // with the static arrays below the 48 KB a launch has unasked
    if (n <= (int64_t)64 * ncells) {
        gbms_shift_kernel<128, CAP><<<ncells, 128, CAP * sizeof(float4), s>>>(spts, boxes, ukeys, table, nslots, d, h,
                                                                              max_iter, modes, counts, st);
    } else {
        gbms_shift_kernel<512, CAP><<<ncells, 512, CAP * sizeof(float4), s>>>(spts, boxes, ukeys, table, nslots, d, h,
                                                                              max_iter, modes, counts, st);
    }
    return cudaGetLastError();
}

cudaError_t launch_gbms_rank(void* temp, size_t temp_bytes, const int* counts, int64_t n, int ns, uint64_t* rkeys,
                             uint64_t* rkeys_sorted, int* nlive, cudaStream_t s) {
    gbms_rank_keys_kernel<<<(ns + 255) / 256, 256, 0, s>>>(counts, ns, rkeys, nlive);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    size_t tb = temp_bytes;
    // the sort is stable and the keys are in seed order; counts 1 .. n differ in the low bits of n of
    // their field, where those of a dropped seed are all ones
    int bits = 1;
    while (n >> bits) ++bits;
    return cub::DeviceRadixSort::SortKeys(temp, tb, rkeys, rkeys_sorted, ns, 32, 32 + bits, s);
}

cudaError_t launch_gbms_rank_modes(const uint64_t* rkeys_sorted, const int* nlive, int nmax, const double4* modes,
                                   const int* counts, int d, double h, double4* rmodes, int* rcount, uint64_t* mkeys,
                                   int* midx, int* state, DeviceState* st, cudaStream_t s) {
    gbms_rank_modes_kernel<<<(nmax + 255) / 256, 256, 0, s>>>(rkeys_sorted, nlive, modes, counts, d, h, rmodes,
                                                              rcount, mkeys, midx, state, st);
    return cudaGetLastError();
}

cudaError_t launch_gbms_merge_round(const double4* rmodes, const int* nlive, int nmax, const ulonglong2* table,
                                    const int* midx_sorted, int d, double h, int* state, int* undecided,
                                    cudaStream_t s) {
    gbms_merge_round_kernel<<<(nmax + GB_WARPS - 1) / GB_WARPS, GB_WARPS * 32, 0, s>>>(
        rmodes, nlive, table, gbms_table_slots(nmax), midx_sorted, d, h, state, undecided);
    return cudaGetLastError();
}

cudaError_t launch_gbms_output(void* temp, size_t temp_bytes, const int* state, const int* nlive, int nmax,
                               const double4* rmodes, const int* rcount, int d, int* flags, int* pos,
                               double* modes_out, int* counts_out, cudaStream_t s) {
    gbms_kept_flags_kernel<<<(nmax + 255) / 256, 256, 0, s>>>(state, nlive, nmax, flags);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    size_t tb = temp_bytes;
    e = cub::DeviceScan::ExclusiveSum(temp, tb, flags, pos, nmax, s);
    if (e != cudaSuccess) return e;
    gbms_output_kernel<<<(nmax + 255) / 256, 256, 0, s>>>(flags, pos, nlive, rmodes, rcount, d, modes_out,
                                                          counts_out);
    return cudaGetLastError();
}

}  // namespace gira
