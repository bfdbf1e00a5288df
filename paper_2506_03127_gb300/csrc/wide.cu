// The MACGIC-iQUAPI path update with keys of up to 128 bits: M up to 8
// system states and windows of up to 16 points (the production models of
// Sec. 4.3 need M = 8 at Delta k_max = 12, 72 bits with two 3-bit states per
// point).  A stored key holds one byte per window position (position 0 =
// newest point in the lowest byte): the forward state in the low nibble,
// the backward state in the high one, in two 64-bit words (lo: positions
// 0..7, hi: 8..15).  The order of these keys, as 128-bit numbers, compares
// the oldest position first and the backward state before the forward one:
// the order of the packed keys of the narrow engines, so the tie rule of
// the pre-merge (reading R4) is the same.
//
// One step (Sec. 3.1, Schemes merging and propagation), pre-merging order:
//   k_w_insert  group every stored path by its P' positions (a 64-bit group
//               key of 6 bits per position) in an open-addressing table:
//               FP64 sums, largest weight (Sec. 3.1 "Pre-merging");
//   k_w_tie     members within the tie window of the largest weight compete
//               on a 64-bit tie key (the positions outside P', in key order);
//               the representative's key is its group key and the winning
//               tie key put together again;
//   k_w_expand  the M^2 children of each group (Eqs. SysP, inf_fun), the
//               filter (|amp| >= theta, Sec. 2.1), the output and rho(t) by
//               newest point (Eq. quapi_red_rho);
//   k_w_finalize the step's rho, counts and state.
// While the window fills every stored path is its own group (reading R3).
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <type_traits>
#include <cstdint>
#include <cstring>
#include <string>
#include <vector>

#include "internal.h"

namespace {

constexpr int kWMaxM = 8, kWMaxDk = 16, kWMaxMM = 64;
constexpr int kWThreads = 256;
// Probes before the table counts as full.  Half of the slots in use are
// allowed (max_groups groups, or as many groups as paths in table_slots):
// there the longest probe of n keys is about ln(n) / 0.19, 72 at 1e6 and 103
// at 4e8 (79 met with 1.7e7), and none reaches 1024; every kWProbeCheck probes
// a path asks whether the step has failed, so that more groups than the table
// holds end soon.
constexpr int kWProbe = 1024, kWProbeCheck = 64;
constexpr int kWMaxRuns = 16;       // runs of consecutive positions, each within one word of eight
constexpr int kWMaxBlocks = 2048;   // blocks of the expansion (partials of rho)
constexpr unsigned long long kWEmpty = ~0ull;
constexpr unsigned kWErrPaths = 1u, kWErrGroups = 2u, kWErrProbe = 4u;

struct WState {
    unsigned long long t, n_cur;       // stored set Omega(t) and its size
    unsigned long long n_groups;       // groups of the running step
    unsigned long long n_out;          // children appended by the running step
    unsigned int err;                  // sticky error bits
    unsigned int pad;
};

struct WRec { long long t, groups, extended, kept, inter; };

// a merge-table slot: group key, largest weight (FP64 bits) and the FP64
// sum in one 32-byte sector
struct __align__(32) WSlot {
    unsigned long long gk, wm;
    double sre, sim;
};

// A set of window positions as runs of consecutive ones: run r takes the
// bits mask[r] of word word[r] (compacted to 6 bits per position, eight
// positions per word) from shift[r] to off[r] of the packed key.
struct WRuns {
    int n, npos;
    unsigned char word[kWMaxRuns], shift[kWMaxRuns], off[kWMaxRuns];
    unsigned long long mask[kWMaxRuns];
};

struct WParams {
    int M, dkmax, c64, rho_hist;
    long long max_paths, max_groups;
    unsigned long long tcap;           // slots of the merge table
    WRuns pp, co;                      // positions of P' and of its complement
    double theta2, tie_rel;
    float theta2f;
    double q[kWMaxM];
    float dq2[kWMaxMM];                // -2 log2(e) (q_a - q_b) of child (a, b)
    float log2_theta2;                 // log2 theta^2; -inf: no bound is taken (see k_w_expand)
    unsigned long long *klo[2], *khi[2];
    void *amps[2];
    unsigned int *slot_of, *groups;
    WSlot *slots;
    unsigned long long *ttie;
    const double2 *lut;                // [dkmax][dkmax - 1][256] FP64 history tables
    const float2 *lutf, *lutlo;        // FP32 hi part and residual
    const double2 *w;                  // [M*M child][M*M parent newest]
    const float4 *wf;                  // FP32 hi/lo pairs of w
    const float *lw;                   // [M*M parent][M*M child] log2 |w|^2
    double2 *rho_part;                 // [blocks][M*M]
    double2 *rho_ring;                 // [rho_hist][M*M]
    WRec *stats;                       // [rho_hist]
    WState *st;
};

__device__ __forceinline__ unsigned key_byte(unsigned long long lo, unsigned long long hi, int j) {
    return (unsigned)((j < 8 ? lo >> (8 * j) : hi >> (8 * (j - 8))) & 0xffull);
}
// Eight positions of a key word (one byte each) as 6-bit codes (forward |
// backward << 3), and back.
__device__ __forceinline__ unsigned long long compact6(unsigned long long x) {
    x = (x & 0x0707070707070707ull) | ((x >> 1) & 0x3838383838383838ull);
    x = (x & 0x003f003f003f003full) | ((x & 0x3f003f003f003f00ull) >> 2);
    x = (x & 0x00000fff00000fffull) | ((x & 0x0fff00000fff0000ull) >> 4);
    return (x & 0xffffffull) | ((x >> 8) & 0xffffff000000ull);
}
__device__ __forceinline__ unsigned long long expand6(unsigned long long x) {
    x = (x & 0xffffffull) | ((x & 0xffffff000000ull) << 8);
    x = (x & 0x00000fff00000fffull) | ((x & 0x00fff00000fff000ull) << 4);
    x = (x & 0x003f003f003f003full) | ((x & 0x0fc00fc00fc00fc0ull) << 2);
    return (x & 0x0707070707070707ull) | ((x & 0x3838383838383838ull) << 1);
}
// The codes of a set of positions packed in ascending order: equal on P' <=>
// equal group keys; on the complement the order of the full keys.
__device__ __forceinline__ unsigned long long pack_runs(const WRuns &R, unsigned long long c0, unsigned long long c1) {
    unsigned long long k = 0;
    for (int r = 0; r < R.n; ++r) k |= (((R.word[r] ? c1 : c0) >> R.shift[r]) & R.mask[r]) << R.off[r];
    return k;
}
__device__ __forceinline__ void unpack_runs(const WRuns &R, unsigned long long k, unsigned long long &c0,
                                            unsigned long long &c1) {
    for (int r = 0; r < R.n; ++r) {
        const unsigned long long v = ((k >> R.off[r]) & R.mask[r]) << R.shift[r];
        if (R.word[r]) c1 |= v;
        else c0 |= v;
    }
}
__device__ __forceinline__ unsigned long long wmix(unsigned long long x) {
    x ^= x >> 31;
    x *= 0x7fb5d329728ea185ull;
    x ^= x >> 27;
    x *= 0x81dadef4bc2dd44dull;
    x ^= x >> 33;
    return x;
}
// s + e += b with the rounding error of the addition carried into e (TwoSum)
__device__ __forceinline__ void two_sum_w(float &s, float &e, float b) {
    const float t = s + b, v = t - s;
    e += (s - (t - v)) + (b - v);
    s = t;
}
__device__ __forceinline__ double weight_of(const WParams &P, const void *amps, unsigned long long i) {
    if (P.c64) {
        const float2 a = static_cast<const float2 *>(amps)[i];
        return (double)(a.x * a.x + a.y * a.y);
    }
    const double2 a = static_cast<const double2 *>(amps)[i];
    return a.x * a.x + a.y * a.y;
}
__device__ __forceinline__ double2 amp_of(const WParams &P, const void *amps, unsigned long long i) {
    if (P.c64) {
        const float2 a = static_cast<const float2 *>(amps)[i];
        return make_double2(a.x, a.y);
    }
    return static_cast<const double2 *>(amps)[i];
}

// Whether the propagation has failed, the same answer for every thread of the
// block: other blocks of a kernel may raise the error while this one reads it,
// and threads that left alone would leave the others' shared scans without
// their part.  Every thread of the block calls it.
__device__ __forceinline__ bool failed_block(const WState *st) {
    return __syncthreads_or(st->err != 0u) != 0;
}

// The part of the table that a step of n paths uses: two slots per path at
// most (at least a page), so that a small step stays near the L2.
__device__ __forceinline__ unsigned long long table_slots(const WParams &P, unsigned long long n) {
    return min(P.tcap, max(2ull * n, 1024ull));
}

// pre-merge, pass 1: claim or find the group's slot, add the amplitude,
// raise the largest weight; the new groups of a block's round are listed with
// one atomic.  Bound: the latency of a random 32-byte slot per path.
__global__ void __launch_bounds__(kWThreads) k_w_insert(WParams P) {
    __shared__ unsigned s_wc[kWThreads / 32];
    __shared__ unsigned long long s_base;
    WState *st = P.st;
    if (failed_block(st)) return;
    const int in = (int)(st->t & 1);
    const unsigned long long n = st->n_cur, slots = table_slots(P, n);
    const unsigned lane = threadIdx.x & 31u, warp = threadIdx.x >> 5;
    for (unsigned long long base = blockIdx.x * (unsigned long long)kWThreads; base < n;
         base += (unsigned long long)gridDim.x * kWThreads) {
        const unsigned long long i = base + threadIdx.x;
        bool claimed = false;
        unsigned long long h = 0;
        if (i < n) {
            const unsigned long long lo = P.klo[in][i], hi = P.khi[in][i];
            const unsigned long long gk = pack_runs(P.pp, compact6(lo), compact6(hi));
            const double2 a = amp_of(P, P.amps[in], i);
            h = __umul64hi(wmix(gk), slots);
            int probe = 0;
            for (; probe < kWProbe; ++probe, h = h + 1 == slots ? 0 : h + 1) {
                unsigned long long cur = *(volatile unsigned long long *)&P.slots[h].gk;
                if (cur == kWEmpty) {
                    cur = atomicCAS(&P.slots[h].gk, kWEmpty, gk);
                    if (cur == kWEmpty) {   // a new group
                        claimed = true;
                        break;
                    }
                }
                if (cur == gk) break;
                if (probe % kWProbeCheck == kWProbeCheck - 1 && *(volatile unsigned *)&st->err) probe = kWProbe - 1;
            }
            if (probe == kWProbe) {
                atomicOr(&st->err, kWErrProbe);
            } else {
                atomicAdd(&P.slots[h].sre, a.x);
                atomicAdd(&P.slots[h].sim, a.y);
                atomicMax(&P.slots[h].wm, (unsigned long long)__double_as_longlong(weight_of(P, P.amps[in], i)));
                P.slot_of[i] = (unsigned)h;
            }
        }
        const unsigned cm = __ballot_sync(0xffffffffu, claimed);
        if (lane == 0) s_wc[warp] = __popc(cm);
        __syncthreads();
        if (threadIdx.x == 0) {
            unsigned tot = 0;
            for (int w = 0; w < kWThreads / 32; ++w) {
                const unsigned v = s_wc[w];
                s_wc[w] = tot;
                tot += v;
            }
            s_base = tot ? atomicAdd(&st->n_groups, (unsigned long long)tot) : 0ull;
        }
        __syncthreads();
        if (claimed) {
            const unsigned long long g = s_base + s_wc[warp] + __popc(cm & ((1u << lane) - 1u));
            if (g < (unsigned long long)P.max_groups) P.groups[g] = (unsigned)h;
            else atomicOr(&st->err, kWErrGroups);
        }
        __syncthreads();   // s_wc and s_base are rewritten in the next round
    }
}

// pre-merge, pass 2: members within the tie window compete on the tie key
__global__ void __launch_bounds__(kWThreads) k_w_tie(WParams P) {
    WState *st = P.st;
    if (st->err) return;
    const int in = (int)(st->t & 1);
    const unsigned long long n = st->n_cur;
    for (unsigned long long i = blockIdx.x * (unsigned long long)blockDim.x + threadIdx.x; i < n;
         i += (unsigned long long)gridDim.x * blockDim.x) {
        const unsigned h = P.slot_of[i];
        const double wm = __longlong_as_double((long long)P.slots[h].wm);
        if (weight_of(P, P.amps[in], i) < (1.0 - P.tie_rel) * wm) continue;
        atomicMin(&P.ttie[h], pack_runs(P.co, compact6(P.klo[in][i]), compact6(P.khi[in][i])));
    }
}

// log2 of a square to FP32 accuracy, off the FP64 pipe, never below it by more
// than that: zero and subnormals, which a square may have underflowed to, give
// -1022, infinities and NaNs +inf, which no bound drops
__device__ __forceinline__ float log2_d(double d) {
    const unsigned long long u = (unsigned long long)__double_as_longlong(d);
    const int e = (int)((u >> 52) & 0x7ffull);
    if (e == 0) return -1022.f;
    if (e == 0x7ff) return INFINITY;
    return (float)(e - 1023) + log2f(__uint_as_float(0x3f800000u | (unsigned)((u >> 29) & 0x7fffffull)));
}

inline size_t expand_smem(int MM, int nb, bool c64) {
    const size_t ct = c64 ? 8 : 16, lw = (size_t)MM * ((MM + 7) & ~3) * 4;
    return (size_t)nb * 64 * 16 + (size_t)(kWThreads / 32) * MM * (c64 ? 24 : 16) + 2 * kWThreads * ct + 2 * kWThreads * 8 +
           ((lw + 15) & ~(size_t)15) + (size_t)MM * (kWThreads / 32) * 8 + kWThreads + (size_t)kWThreads * MM * 2;
}

// The children of the step's groups (merge) or stored paths (window filling).
// A block takes 256 groups per round.  With most of the M^2 children below
// the filter (the reaction-coordinate model keeps about 2 of 64) each thread
// first bounds the 64 weights of its group,
//   log2 |child|^2 = log2 |S|^2 + log2 |W|^2 - 2 log2(e) (q_a - q_b) Re H,
// one table entry, one multiply-add and one comparison per child in FP32,
// with a margin of 2^0.002 (the terms are good to about 2^-16); the children
// above the bound are listed child-major for the block, so that they are
// dealt evenly to the threads and a warp's children share their newest
// point; each is formed once in full precision, filtered, added to rho(t)
// (segments of equal newest point, then one lane's addition to its warp's
// bin; C64: sums of three FP32 words with TwoSum, as close to the exact sum as
// FP64 ones, 1e-16 at most in rho, at 16.8 ms per 20 steps of the eight-state
// model, FP64 17.7 to 17.9; pairs, 16.4 ms, left up to 1e-15) and written to a
// range reserved per 256
// candidates.  (Forming all 64 children twice, four lanes per group, with
// rho from a second pass over the children took 0.88 ms per step and launch
// at 2e6 groups, the two passes of rho and of its block sums 0.30 ms.)
template <bool C64>
__global__ void __launch_bounds__(kWThreads) k_w_expand(WParams P, int merge) {
    using CT = typename std::conditional<C64, float2, double2>::type;
    constexpr int NW = kWThreads / 32;
    extern __shared__ __align__(16) unsigned char s_dyn[];
    __shared__ unsigned s_wc[NW], s_tot;
    __shared__ unsigned long long s_base;
    WState *st = P.st;
    const int M = P.M, MM = M * M;
    const int nb = P.dkmax - 1;                       // history bytes of a key
    const int lws = (MM + 7) & ~3;                    // row of the bound table (rows on different banks)
    float4 *s_lut = reinterpret_cast<float4 *>(s_dyn);   // [nb][64] history terms (C64: hi, lo; FP64: double2)
    float4 *s_rho = s_lut + nb * 64;                     // [NW][MM] (C64: re, err, im, err; FP64: double2)
    float2 *s_rhof = reinterpret_cast<float2 *>(s_rho + NW * MM);   // C64: what is lost of the errors
    CT *s_S = reinterpret_cast<CT *>(s_rhof + (C64 ? NW * MM : 0)), *s_H = s_S + kWThreads;
    unsigned long long *s_lo = reinterpret_cast<unsigned long long *>(s_H + kWThreads), *s_hi = s_lo + kWThreads;
    float *s_lw = reinterpret_cast<float *>(s_hi + kWThreads);
    unsigned *s_mask = reinterpret_cast<unsigned *>(s_lw + ((MM * lws + 3) & ~3));   // [MM][NW] candidates of a warp
    unsigned *s_off = s_mask + MM * NW;                                              // [MM][NW] their offsets
    unsigned char *s_par = reinterpret_cast<unsigned char *>(s_off + MM * NW);
    unsigned short *s_list = reinterpret_cast<unsigned short *>(s_par + kWThreads);
    const unsigned lane = threadIdx.x & 31u, warp = threadIdx.x >> 5;
    double2 *part = P.rho_part + (size_t)blockIdx.x * MM;
    if (failed_block(st)) return;
    const unsigned long long t = st->t, tn = t + 1;
    const int in = (int)(t & 1), outp = (int)(tn & 1);
    const unsigned long long ng = merge ? st->n_groups : st->n_cur;
    const int n_act = (int)min(tn, (unsigned long long)P.dkmax);
    const int L_child = (int)min(tn + 1, (unsigned long long)P.dkmax);
    const size_t row = (size_t)(n_act - 1) * nb * 256;
    for (int i = threadIdx.x; i < nb * 64; i += kWThreads) {
        const size_t j = row + (size_t)(i >> 6) * 256 + ((i & 7) | ((i & 56) << 1));
        if constexpr (C64) {
            const float2 a = P.lutf[j], b = P.lutlo[j];
            s_lut[i] = make_float4(a.x, a.y, b.x, b.y);
        } else {
            reinterpret_cast<double2 *>(s_lut)[i] = P.lut[j];
        }
    }
    for (int i = threadIdx.x; i < MM * lws; i += kWThreads)
        s_lw[i] = i % lws < MM ? P.lw[(size_t)(i / lws) * MM + i % lws] : -INFINITY;
    for (int i = threadIdx.x; i < NW * MM; i += kWThreads) {
        s_rho[i] = make_float4(0.f, 0.f, 0.f, 0.f);
        if constexpr (C64) s_rhof[i] = make_float2(0.f, 0.f);
    }
    __syncthreads();
    for (unsigned long long base = blockIdx.x * (unsigned long long)kWThreads; base < ng;
         base += (unsigned long long)gridDim.x * kWThreads) {
        const unsigned long long g = base + threadIdx.x;
        const bool valid = g < ng;
        float thr = INFINITY, hre = 0.f;   // a child is a candidate unless its bound is below thr
        int parc = 0;
        if (valid) {
            unsigned long long lo, hi;
            double2 S;
            if (merge) {
                const unsigned h = P.groups[g];
                const WSlot sl = P.slots[h];
                S = make_double2(sl.sre, sl.sim);
                unsigned long long c0 = 0, c1 = 0;
                unpack_runs(P.pp, sl.gk, c0, c1);
                unpack_runs(P.co, P.ttie[h], c0, c1);
                lo = expand6(c0);
                hi = expand6(c1);
                WSlot fresh;   // the slot is this group's: free for the next step
                fresh.gk = kWEmpty;
                fresh.wm = 0ull;
                fresh.sre = fresh.sim = 0.0;
                P.slots[h] = fresh;
                P.ttie[h] = kWEmpty;
            } else {
                S = amp_of(P, P.amps[in], g);
                lo = P.klo[in][g];
                hi = P.khi[in][g];
            }
            const int par = (int)(lo & 0xffull);
            parc = (par & 15) * M + (par >> 4);   // (forward, backward) of the newest point
            // history part H of the influence exponent: FP64, or FP32 with the
            // rounding of every addition kept (Kahan) from the hi/lo tables
            if constexpr (C64) {
                float hx = 0.f, hy = 0.f, cx = 0.f, cy = 0.f;
                for (int j = 0; j < nb; ++j) {
                    const unsigned v = key_byte(lo, hi, j);
                    const float4 e = s_lut[j * 64 + ((v & 7u) | ((v >> 1) & 56u))];
                    float yx = (e.x - cx), tx = hx + yx;
                    cx = (tx - hx) - yx;
                    hx = tx;
                    yx = (e.z - cx);
                    tx = hx + yx;
                    cx = (tx - hx) - yx;
                    hx = tx;
                    float yy = (e.y - cy), ty = hy + yy;
                    cy = (ty - hy) - yy;
                    hy = ty;
                    yy = (e.w - cy);
                    ty = hy + yy;
                    cy = (ty - hy) - yy;
                    hy = ty;
                }
                s_H[threadIdx.x] = make_float2(hx, hy);
                s_S[threadIdx.x] = make_float2((float)S.x, (float)S.y);
                hre = hx;
            } else {
                double Hx = 0.0, Hy = 0.0;
                for (int j = 0; j < nb; ++j) {
                    const unsigned v = key_byte(lo, hi, j);
                    const double2 e = reinterpret_cast<const double2 *>(s_lut)[j * 64 + ((v & 7u) | ((v >> 1) & 56u))];
                    Hx += e.x;
                    Hy += e.y;
                }
                s_H[threadIdx.x] = make_double2(Hx, Hy);
                s_S[threadIdx.x] = S;
                hre = (float)Hx;
            }
            thr = P.log2_theta2 == -INFINITY ? -INFINITY : P.log2_theta2 - 0.002f - log2_d(S.x * S.x + S.y * S.y);
            // child key: the parent shifted up one position, the new point in
            // the lowest byte, cut to L_child positions
            unsigned long long chi = (hi << 8) | (lo >> 56), clo = lo << 8;
            if (8 * L_child <= 64) {
                chi = 0;
                if (8 * L_child < 64) clo &= (1ull << (8 * L_child)) - 1ull;
            } else if (8 * L_child < 128) {
                chi &= (1ull << (8 * L_child - 64)) - 1ull;
            }
            s_lo[threadIdx.x] = clo;
            s_hi[threadIdx.x] = chi;
            s_par[threadIdx.x] = (unsigned char)parc;
        }
        // the candidates of each child as warp masks
        unsigned long long mine = 0ull;
        for (int c0 = 0; c0 < MM; c0 += 4) {
            const float4 l4 = *reinterpret_cast<const float4 *>(s_lw + parc * lws + c0);
            const float lv[4] = {l4.x, l4.y, l4.z, l4.w};
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                const int c = c0 + u;
                if (c >= MM) break;
                const bool cand = valid && !(fmaf(P.dq2[c], hre, lv[u]) < thr);
                const unsigned m = __ballot_sync(0xffffffffu, cand);
                if (cand) mine |= 1ull << c;
                if (lane == 0) s_mask[c * NW + warp] = m;
            }
        }
        __syncthreads();
        {   // exclusive scan of the MM * NW counts, two per thread
            const int i0 = 2 * (int)threadIdx.x;
            const unsigned n0 = i0 < MM * NW ? __popc(s_mask[i0]) : 0u, n1 = i0 + 1 < MM * NW ? __popc(s_mask[i0 + 1]) : 0u;
            unsigned inc = n0 + n1;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const unsigned y = __shfl_up_sync(0xffffffffu, inc, o);
                if ((int)lane >= o) inc += y;
            }
            if (lane == 31) s_wc[warp] = inc;
            __syncthreads();
            unsigned before = 0;
            for (int w = 0; w < NW; ++w)
                if (w < (int)warp) before += s_wc[w];
            const unsigned ex = before + inc - n0 - n1;
            if (i0 < MM * NW) s_off[i0] = ex;
            if (i0 + 1 < MM * NW) s_off[i0 + 1] = ex + n0;
            if (threadIdx.x == kWThreads - 1) s_tot = ex + n0 + n1;
        }
        __syncthreads();
        for (unsigned long long m = mine; m; m &= m - 1ull) {
            const int c = __ffsll((long long)m) - 1, q = c * NW + (int)warp;
            s_list[s_off[q] + __popc(s_mask[q] & ((1u << lane) - 1u))] = (unsigned short)(threadIdx.x | (c << 8));
        }
        __syncthreads();
        const unsigned total = s_tot;
        for (unsigned p0 = 0; p0 < total; p0 += kWThreads) {
            const unsigned p = p0 + threadIdx.x;
            const bool have = p < total;
            const unsigned e = have ? s_list[p] : 0u;
            const int c = have ? (int)(e >> 8) : 0xff, src = (int)(e & 0xffu);
            bool kept = false;
            CT child;
            child.x = child.y = 0;
            int code = 0;
            if (have) {
                const int a = c / M, b = c - a * M;
                code = a | (b << 4);
                const double dq = P.q[a] - P.q[b];
                const CT H = s_H[src], S = s_S[src];
                if constexpr (C64) {
                    float fx = 1.f, fy = 0.f;
                    if (dq != 0.0) {
                        const float dqf = (float)dq;
                        const float zr = -dqf * H.x, zi = -dqf * H.y;
                        float sn, cs;
                        sincosf(zi, &sn, &cs);
                        const float m = expf(zr);
                        fx = m * cs;
                        fy = m * sn;
                    }
                    const float4 wv = P.wf[(size_t)c * MM + s_par[src]];
                    // S (W_hi + W_lo) f
                    const float px = fmaf(S.x, wv.x, -S.y * wv.y) + fmaf(S.x, wv.z, -S.y * wv.w);
                    const float py = fmaf(S.x, wv.y, S.y * wv.x) + fmaf(S.x, wv.w, S.y * wv.z);
                    child = make_float2(px * fx - py * fy, px * fy + py * fx);
                    kept = child.x * child.x + child.y * child.y >= P.theta2f;
                } else {
                    double fx = 1.0, fy = 0.0;
                    if (dq != 0.0) {
                        const double zr = -dq * H.x, zi = -dq * H.y;
                        double sn, cs;
                        sincos(zi, &sn, &cs);
                        const double m = exp(zr);
                        fx = m * cs;
                        fy = m * sn;
                    }
                    const double2 wv = P.w[(size_t)c * MM + s_par[src]];
                    const double px = S.x * wv.x - S.y * wv.y, py = S.x * wv.y + S.y * wv.x;
                    child = make_double2(px * fx - py * fy, px * fy + py * fx);
                    kept = child.x * child.x + child.y * child.y >= P.theta2;
                }
            }
            // rho(t+1): the kept children of a segment of equal c, added by
            // its last lane to the warp's bin
            {
                CT s = child, er, ef;   // C64: three words
                er.x = er.y = ef.x = ef.y = 0;
                if (!kept) s.x = s.y = 0;
#pragma unroll
                for (int o = 1; o < 32; o <<= 1) {
                    const int cu = __shfl_up_sync(0xffffffffu, c, o);
                    const bool add = (int)lane >= o && cu == c;
                    if constexpr (C64) {
                        const float bx = __shfl_up_sync(0xffffffffu, s.x, o), by = __shfl_up_sync(0xffffffffu, s.y, o);
                        float ex = 0.f, ey = 0.f, fx = 0.f, fy = 0.f;   // (the words that are there after o = 1, 2)
                        if (o > 1) {
                            ex = __shfl_up_sync(0xffffffffu, er.x, o);
                            ey = __shfl_up_sync(0xffffffffu, er.y, o);
                        }
                        if (o > 2) {
                            fx = __shfl_up_sync(0xffffffffu, ef.x, o);
                            fy = __shfl_up_sync(0xffffffffu, ef.y, o);
                        }
                        if (add) {
                            float gx = 0.f, gy = 0.f;
                            two_sum_w(s.x, gx, bx);
                            two_sum_w(s.y, gy, by);
                            if (o == 1) {
                                er.x = gx;
                                er.y = gy;
                            } else {
                                two_sum_w(er.x, ef.x, gx);
                                two_sum_w(er.y, ef.y, gy);
                                two_sum_w(er.x, ef.x, ex);
                                two_sum_w(er.y, ef.y, ey);
                                ef.x += fx;
                                ef.y += fy;
                            }
                        }
                    } else {
                        const double bx = __shfl_up_sync(0xffffffffu, s.x, o), by = __shfl_up_sync(0xffffffffu, s.y, o);
                        if (add) {
                            s.x += bx;
                            s.y += by;
                        }
                    }
                }
                const int cn = __shfl_down_sync(0xffffffffu, c, 1);
                if (have && (lane == 31u || cn != c)) {
                    float4 &bin = s_rho[warp * MM + c];
                    if constexpr (C64) {
                        float4 v = bin;
                        float2 f = s_rhof[warp * MM + c];
                        float gx = 0.f, gy = 0.f;
                        two_sum_w(v.x, gx, s.x);
                        two_sum_w(v.z, gy, s.y);
                        two_sum_w(v.y, f.x, gx);
                        two_sum_w(v.w, f.y, gy);
                        two_sum_w(v.y, f.x, er.x);
                        two_sum_w(v.w, f.y, er.y);
                        f.x += ef.x;
                        f.y += ef.y;
                        bin = v;
                        s_rhof[warp * MM + c] = f;
                    } else {
                        double2 v = reinterpret_cast<double2 &>(bin);
                        v.x += s.x;
                        v.y += s.y;
                        reinterpret_cast<double2 &>(bin) = v;
                    }
                }
            }
            const unsigned km = __ballot_sync(0xffffffffu, kept);
            if (lane == 0) s_wc[warp] = __popc(km);
            __syncthreads();
            if (threadIdx.x == 0) {
                unsigned tot = 0;
                for (int w = 0; w < NW; ++w) {
                    const unsigned v = s_wc[w];
                    s_wc[w] = tot;
                    tot += v;
                }
                s_base = tot ? atomicAdd(&st->n_out, (unsigned long long)tot) : 0ull;
            }
            __syncthreads();
            if (kept) {
                const unsigned long long o = s_base + s_wc[warp] + __popc(km & ((1u << lane) - 1u));
                if (o >= (unsigned long long)P.max_paths) {
                    atomicOr(&st->err, kWErrPaths);
                } else {
                    P.klo[outp][o] = s_lo[src] | (unsigned long long)code;
                    P.khi[outp][o] = s_hi[src];
                    static_cast<CT *>(P.amps[outp])[o] = child;
                }
            }
            __syncthreads();   // s_wc and s_base are rewritten
        }
        // (the loop's last barrier, or none of its shared arrays read: the
        // next round may overwrite them)
        __syncthreads();
    }
    // this block's sums of rho, the warps in order
    for (int k = threadIdx.x; k < MM; k += kWThreads) {
        if constexpr (C64) {
            double2 v = make_double2(0.0, 0.0);
            for (int w = 0; w < NW; ++w) {
                const float4 b = s_rho[w * MM + k];
                const float2 f = s_rhof[w * MM + k];
                // (the errors of an infinite sum are not numbers)
                v.x += isfinite(b.x) ? (double)b.x + ((double)b.y + (double)f.x) : (double)b.x;
                v.y += isfinite(b.z) ? (double)b.z + ((double)b.w + (double)f.y) : (double)b.z;
            }
            part[k] = v;
        } else {
            double2 v = reinterpret_cast<const double2 *>(s_rho)[k];
            for (int w = 1; w < NW; ++w) {
                const double2 b = reinterpret_cast<const double2 *>(s_rho)[w * MM + k];
                v.x += b.x;
                v.y += b.y;
            }
            part[k] = v;
        }
    }
}

// one block of 1024 threads: rho(t+1) from the block sums (1024 / M^2 threads
// per component, then in order), the step's record, the new state
__global__ void __launch_bounds__(1024) k_w_finalize(WParams P, int nblk, int merge) {
    __shared__ double2 s_p[1024];
    WState *st = P.st;
    const int MM = P.M * P.M;
    if (st->err) return;
    const unsigned long long tn = st->t + 1;
    const size_t slot = (size_t)(tn % (unsigned long long)P.rho_hist);
    const int T = 1024 / MM, k = (int)threadIdx.x % MM, j = (int)threadIdx.x / MM;
    double x = 0.0, y = 0.0;
    if (j < T)
#pragma unroll 8
        for (int b = j; b < nblk; b += T) {
            const double2 v = P.rho_part[(size_t)b * MM + k];
            x += v.x;
            y += v.y;
        }
    s_p[threadIdx.x] = make_double2(x, y);
    __syncthreads();
    if ((int)threadIdx.x < MM) {
        for (int u = 1; u < T; ++u) {
            x += s_p[u * MM + threadIdx.x].x;
            y += s_p[u * MM + threadIdx.x].y;
        }
        P.rho_ring[slot * MM + threadIdx.x] = make_double2(x, y);
    }
    if (threadIdx.x == 0) {
        const unsigned long long groups = merge ? st->n_groups : st->n_cur;
        WRec r;
        r.t = (long long)tn;
        r.groups = (long long)groups;
        r.extended = (long long)groups * MM;
        r.kept = (long long)st->n_out;
        r.inter = r.kept;
        P.stats[slot] = r;
        st->n_cur = st->n_out;
        st->t = tn;
        st->n_groups = 0;
        st->n_out = 0;
    }
}

// history tables: T[n_act][j][v] = eta_{j+1} q[forward] - conj(eta_{j+1})
// q[backward] for the point at byte j of a key while n_act points are held
// (bytes past the history contribute nothing)
__global__ void k_w_build_lut(double2 *lut, float2 *lutf, float2 *lutlo, const double2 *eta, const double *q, int M,
                              int dkmax) {
    const int nb = dkmax - 1, total = dkmax * nb * 256;
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < total; i += gridDim.x * blockDim.x) {
        const int v = i % 256, j = (i / 256) % nb, n_act = i / (256 * nb) + 1;
        const int sp = v & 15, sm = v >> 4;
        double hx = 0.0, hy = 0.0;
        if (j <= n_act - 2 && sp < M && sm < M) {
            const double2 e = eta[j + 1];
            hx = e.x * q[sp] - e.x * q[sm];
            hy = e.y * q[sp] + e.y * q[sm];
        }
        lut[i] = make_double2(hx, hy);
        const float fx = (float)hx, fy = (float)hy;
        lutf[i] = make_float2(fx, fy);
        lutlo[i] = make_float2((float)(hx - (double)fx), (float)(hy - (double)fy));
    }
}

// W[(a,b)][(a',b')] = U[a,a'] conj(U[b,b']) exp(-(q_a - q_b)(eta_0 q_a - conj(eta_0) q_b))
__global__ void k_w_build_w(double2 *w, float4 *wf, float *lw, const double2 *U, const double2 *eta, const double *q, int M) {
    const int MM = M * M;
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < MM * MM; i += gridDim.x * blockDim.x) {
        const int child = i / MM, par = i % MM;
        const int a = child / M, b = child % M, ap = par / M, bp = par % M;
        const double2 ua = U[a * M + ap], ub = U[b * M + bp];
        const double2 prop = make_double2(ua.x * ub.x + ua.y * ub.y, ua.y * ub.x - ua.x * ub.y);
        const double dq = q[a] - q[b];
        const double2 e0 = eta[0];
        const double zr = -dq * (e0.x * q[a] - e0.x * q[b]), zi = -dq * (e0.y * q[a] + e0.y * q[b]);
        double s, c;
        sincos(zi, &s, &c);
        const double m = exp(zr);
        const double2 f = make_double2(m * c, m * s);
        const double2 v = make_double2(prop.x * f.x - prop.y * f.y, prop.x * f.y + prop.y * f.x);
        w[i] = v;
        const float hx = (float)v.x, hy = (float)v.y;
        wf[i] = make_float4(hx, hy, (float)(v.x - (double)hx), (float)(v.y - (double)hy));
        lw[(size_t)par * MM + child] = (float)(2.0 * log2(hypot(v.x, v.y)));   // (no square to underflow)
    }
}

__global__ void k_w_clear_table(WSlot *slots, unsigned long long *ttie, unsigned long long n) {
    for (unsigned long long i = blockIdx.x * (unsigned long long)blockDim.x + threadIdx.x; i < n;
         i += (unsigned long long)gridDim.x * blockDim.x) {
        WSlot fresh;
        fresh.gk = kWEmpty;
        fresh.wm = 0ull;
        fresh.sre = fresh.sim = 0.0;
        slots[i] = fresh;
        ttie[i] = kWEmpty;
    }
}

size_t a256(size_t x) { return (x + 255) & ~(size_t)255; }

struct WLayout {
    size_t klo[2], khi[2], amps[2], slot_of, groups, slots, ttie, lut, lutf, lutlo, w, wf, lw, U, eta, q,
        rho_part, rho, stats, state, total;
    unsigned long long tcap;
};

const char *wide_invalid(const qp_config *c) {
    if (!c) return "null config";
    if (c->M < 2 || c->M > kWMaxM) return "M out of range (2..8)";
    if (c->dkmax < 1 || c->dkmax > kWMaxDk) return "dkmax out of range (1..16)";
    if (!(c->dt > 0.0) || !std::isfinite(c->dt)) return "dt must be positive";
    if (!(c->theta >= 0.0) || !std::isfinite(c->theta)) return "theta must be >= 0";
    if (c->precision != QP_FP64 && c->precision != QP_C64) return "unknown precision";
    if (c->max_paths < 16 || c->max_paths > (1ll << 32)) return "max_paths out of range (16 .. 2^32)";
    if (c->max_groups < 0 || c->max_groups > (1ll << 32)) return "max_groups out of range";
    if (c->rho_history < 0 || c->rho_history > (1 << 20)) return "rho_history out of range";
    if (c->n_inst > 1) return "wide keys take single problems only";
    if (c->scheme != QP_PREMERGE) return "wide keys take the pre-merging order only";
    if (!c->q || !c->hs_re) return "q and hs required";
    for (int i = 0; i < c->M; ++i)
        if (!std::isfinite(c->q[i])) return "q must be finite";
    return nullptr;
}

WLayout wide_layout(const qp_config *c) {
    WLayout L{};
    const long long mp = c->max_paths;
    const long long mg = c->max_groups ? c->max_groups : mp;
    unsigned long long tcap = 16;
    while (tcap < 2ull * (unsigned long long)mg) tcap <<= 1;
    L.tcap = tcap;
    const int MM = c->M * c->M, R = c->rho_history ? c->rho_history : 4096;
    const size_t ab = c->precision == QP_C64 ? 8 : 16;
    const size_t nlut = (size_t)c->dkmax * std::max(1, c->dkmax - 1) * 256;
    size_t off = 0;
    auto take = [&](size_t bytes) { size_t o = off; off = a256(off + bytes); return o; };
    L.state = take(sizeof(WState));
    for (int k = 0; k < 2; ++k) {
        L.klo[k] = take(mp * 8);
        L.khi[k] = take(mp * 8);
        L.amps[k] = take(mp * ab);
    }
    L.slot_of = take(mp * 4);
    L.groups = take(mg * 4);
    L.slots = take(tcap * sizeof(WSlot));
    L.ttie = take(tcap * 8);
    L.lut = take(nlut * 16);
    L.lutf = take(nlut * 8);
    L.lutlo = take(nlut * 8);
    L.w = take((size_t)MM * MM * 16);
    L.wf = take((size_t)MM * MM * 16);
    L.lw = take((size_t)MM * MM * 4);
    L.U = take((size_t)MM * 16);
    L.eta = take((size_t)c->dkmax * 16);
    L.q = take((size_t)c->M * 8);
    L.rho_part = take((size_t)kWMaxBlocks * MM * 16);
    L.rho = take((size_t)R * MM * 16);
    L.stats = take((size_t)R * sizeof(WRec));
    L.total = off;
    return L;
}

}  // namespace

struct qp_wide {
    qp_config cfg;
    std::vector<double> q;
    std::vector<qp::cplx> hs, U;
    std::vector<int> mask;
    WLayout L;
    WParams P{};
    char *ws = nullptr;
    cudaStream_t stream = nullptr;
    int nsm = 0, nblk = 0, xblk = 0;   // blocks of the table passes and of the expansion
    size_t xsmem = 0;                  // shared memory of the expansion
    bool have_eta = false, have_state = false, failed = false;
    std::string err;
};

namespace {

qp_status wfail(qp_wide *w, qp_status s, const std::string &msg) {
    if (w) w->err = msg;
    return s;
}
#define QW_CUDA(w, call)                                                                         \
    do {                                                                                         \
        cudaError_t e_ = (call);                                                                 \
        if (e_ != cudaSuccess) return wfail((w), QP_ERR_CUDA, std::string(#call) + ": " + cudaGetErrorString(e_)); \
    } while (0)

qp_status wide_set_mask_params(qp_wide *w, const std::vector<int> &P) {
    const int dk = w->cfg.dkmax;
    std::vector<char> in(dk, 0);
    in[0] = 1;
    for (int p : P)
        if (p >= 1) in[p - 1] = 1;
    int np = 0, nc = 0;
    for (int p = 0; p < dk; ++p) ++(in[p] ? np : nc);
    if (6 * np > 64) return wfail(w, QP_ERR_ARG, "wide keys: P' may hold at most 10 positions (64-bit group key)");
    if (6 * nc > 64) return wfail(w, QP_ERR_ARG, "wide keys: at most 10 positions outside P' (64-bit tie key)");
    for (int side = 0; side < 2; ++side) {   // runs of consecutive positions within a word of eight
        WRuns R{};
        for (int p = 0; p < dk;) {
            if ((bool)in[p] != (side == 0)) {
                ++p;
                continue;
            }
            int e = p + 1;
            while (e < dk && (e & 7) && (bool)in[e] == (side == 0)) ++e;
            R.word[R.n] = (unsigned char)(p >> 3);
            R.shift[R.n] = (unsigned char)(6 * (p & 7));
            R.off[R.n] = (unsigned char)(6 * R.npos);
            R.mask[R.n] = (1ull << (6 * (e - p))) - 1ull;
            ++R.n;
            R.npos += e - p;
            p = e;
        }
        (side == 0 ? w->P.pp : w->P.co) = R;
    }
    return QP_OK;
}

qp_status wide_read_state(qp_wide *w, WState *s) {
    QW_CUDA(w, cudaMemcpyAsync(s, w->P.st, sizeof(WState), cudaMemcpyDeviceToHost, w->stream));
    QW_CUDA(w, cudaStreamSynchronize(w->stream));
    if (s->err) {
        w->failed = true;
        std::string what;
        if (s->err & kWErrPaths) what += " path buffer (max_paths)";
        if (s->err & kWErrGroups) what += " merge groups (max_groups)";
        if (s->err & kWErrProbe) what += " merge table probe limit";
        return wfail(w, QP_ERR_CAPACITY, "capacity exceeded at step " + std::to_string(s->t + 1) + ":" + what);
    }
    return QP_OK;
}

}  // namespace

extern "C" {

qp_status qp_wide_workspace_size(const qp_config *cfg, size_t *bytes) {
    if (!bytes || wide_invalid(cfg)) return QP_ERR_ARG;
    *bytes = wide_layout(cfg).total;
    return QP_OK;
}

qp_status qp_wide_create(const qp_config *cfg, void *d_workspace, size_t bytes, void *cuda_stream, qp_wide **out) {
    if (!out) return QP_ERR_ARG;
    *out = nullptr;
    if (wide_invalid(cfg) || !d_workspace) return QP_ERR_ARG;
    const WLayout L = wide_layout(cfg);
    if (bytes < L.total) return QP_ERR_OOM;
    qp_wide *w = new (std::nothrow) qp_wide;
    if (!w) return QP_ERR_OOM;
    w->cfg = *cfg;
    w->q.assign(cfg->q, cfg->q + cfg->M);
    const int M = cfg->M, MM = M * M;
    w->hs.resize(MM);
    for (int i = 0; i < MM; ++i) w->hs[i] = qp::cplx(cfg->hs_re[i], cfg->hs_im ? cfg->hs_im[i] : 0.0);
    w->cfg.q = nullptr;
    w->cfg.hs_re = w->cfg.hs_im = nullptr;
    w->U = qp::short_time_propagator(M, w->hs, cfg->dt);
    w->L = L;
    w->ws = static_cast<char *>(d_workspace);
    w->stream = static_cast<cudaStream_t>(cuda_stream);
    int dev = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&w->nsm, cudaDevAttrMultiProcessorCount, dev);
    w->nblk = std::max(1, w->nsm) * 8;
    WParams &P = w->P;
    P.M = M;
    P.dkmax = cfg->dkmax;
    P.c64 = cfg->precision == QP_C64 ? 1 : 0;
    P.rho_hist = cfg->rho_history ? cfg->rho_history : 4096;
    P.max_paths = cfg->max_paths;
    P.max_groups = cfg->max_groups ? cfg->max_groups : cfg->max_paths;
    P.tcap = L.tcap;
    P.theta2 = cfg->theta * cfg->theta;
    P.theta2f = (float)P.theta2;
    P.tie_rel = cfg->precision == QP_C64 ? 1e-6 : 1e-12;   // the narrow engines' windows (reading R4, R11)
    for (int i = 0; i < M; ++i) P.q[i] = cfg->q[i];
    for (int a = 0; a < M; ++a)
        for (int b = 0; b < M; ++b) P.dq2[a * M + b] = (float)(-2.0 * 1.4426950408889634 * (cfg->q[a] - cfg->q[b]));
    // no filter, or one in the range where squares lose precision to
    // underflow: every child is formed
    P.log2_theta2 = P.theta2 > (P.c64 ? 1e-36 : 1e-290) ? (float)std::log2(P.theta2) : -INFINITY;
    char *ws = w->ws;
    for (int k = 0; k < 2; ++k) {
        P.klo[k] = reinterpret_cast<unsigned long long *>(ws + L.klo[k]);
        P.khi[k] = reinterpret_cast<unsigned long long *>(ws + L.khi[k]);
        P.amps[k] = ws + L.amps[k];
    }
    P.slot_of = reinterpret_cast<unsigned *>(ws + L.slot_of);
    P.groups = reinterpret_cast<unsigned *>(ws + L.groups);
    P.slots = reinterpret_cast<WSlot *>(ws + L.slots);
    P.ttie = reinterpret_cast<unsigned long long *>(ws + L.ttie);
    P.lut = reinterpret_cast<const double2 *>(ws + L.lut);
    P.lutf = reinterpret_cast<const float2 *>(ws + L.lutf);
    P.lutlo = reinterpret_cast<const float2 *>(ws + L.lutlo);
    P.w = reinterpret_cast<const double2 *>(ws + L.w);
    P.wf = reinterpret_cast<const float4 *>(ws + L.wf);
    P.lw = reinterpret_cast<const float *>(ws + L.lw);
    P.rho_part = reinterpret_cast<double2 *>(ws + L.rho_part);
    P.rho_ring = reinterpret_cast<double2 *>(ws + L.rho);
    P.stats = reinterpret_cast<WRec *>(ws + L.stats);
    P.st = reinterpret_cast<WState *>(ws + L.state);
    std::vector<int> full(cfg->dkmax);
    for (int p = 0; p < cfg->dkmax; ++p) full[p] = p;
    w->mask = full;
    if (wide_set_mask_params(w, full) != QP_OK && cfg->dkmax > 0) {
        // the full mask of a long window does not fit a 64-bit group key:
        // a mask must be set before qp_wide_set_rho0
        w->P.pp.npos = -1;
    }
    const void *fn = P.c64 ? (const void *)k_w_expand<true> : (const void *)k_w_expand<false>;
    w->xsmem = expand_smem(MM, cfg->dkmax - 1, P.c64 != 0);
    int res = 0;
    if (cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             (int)expand_smem(kWMaxMM, kWMaxDk - 1, P.c64 != 0)) != cudaSuccess ||
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&res, fn, kWThreads, w->xsmem) != cudaSuccess || res < 1) {
        delete w;
        return QP_ERR_CUDA;
    }
    w->xblk = std::min(kWMaxBlocks, std::max(1, w->nsm) * res);
    *out = w;
    return QP_OK;
}

void qp_wide_destroy(qp_wide *w) { delete w; }

qp_status qp_wide_set_eta(qp_wide *w, const double *re, const double *im, int n) {
    if (!w) return QP_ERR_ARG;
    const int dk = w->cfg.dkmax, M = w->cfg.M, MM = M * M;
    if (!re || !im || n < dk) return wfail(w, QP_ERR_ARG, "need dkmax coefficients");
    std::vector<double2> e(dk), Ud(MM);
    for (int i = 0; i < dk; ++i) {
        if (!std::isfinite(re[i]) || !std::isfinite(im[i])) return wfail(w, QP_ERR_ARG, "eta must be finite");
        e[i] = make_double2(re[i], im[i]);
    }
    for (int i = 0; i < MM; ++i) Ud[i] = make_double2(w->U[i].real(), w->U[i].imag());
    char *ws = w->ws;
    QW_CUDA(w, cudaMemcpyAsync(ws + w->L.eta, e.data(), dk * sizeof(double2), cudaMemcpyHostToDevice, w->stream));
    QW_CUDA(w, cudaMemcpyAsync(ws + w->L.U, Ud.data(), MM * sizeof(double2), cudaMemcpyHostToDevice, w->stream));
    QW_CUDA(w, cudaMemcpyAsync(ws + w->L.q, w->q.data(), M * sizeof(double), cudaMemcpyHostToDevice, w->stream));
    if (dk >= 2)
        k_w_build_lut<<<64, 256, 0, w->stream>>>(reinterpret_cast<double2 *>(ws + w->L.lut),
                                                 reinterpret_cast<float2 *>(ws + w->L.lutf),
                                                 reinterpret_cast<float2 *>(ws + w->L.lutlo),
                                                 reinterpret_cast<const double2 *>(ws + w->L.eta),
                                                 reinterpret_cast<const double *>(ws + w->L.q), M, dk);
    k_w_build_w<<<16, 256, 0, w->stream>>>(reinterpret_cast<double2 *>(ws + w->L.w),
                                           reinterpret_cast<float4 *>(ws + w->L.wf),
                                           reinterpret_cast<float *>(ws + w->L.lw),
                                           reinterpret_cast<const double2 *>(ws + w->L.U),
                                           reinterpret_cast<const double2 *>(ws + w->L.eta),
                                           reinterpret_cast<const double *>(ws + w->L.q), M);
    QW_CUDA(w, cudaGetLastError());
    QW_CUDA(w, cudaStreamSynchronize(w->stream));   // e, Ud are host temporaries
    w->have_eta = true;
    return QP_OK;
}

qp_status qp_wide_set_mask(qp_wide *w, const int *positions, int n) {
    if (!w) return QP_ERR_ARG;
    const int dk = w->cfg.dkmax;
    std::vector<int> P;
    if (!positions || n == 0) {
        for (int p = 0; p < dk; ++p) P.push_back(p);
    } else {
        for (int i = 0; i < n; ++i) {
            if (positions[i] < 0 || positions[i] >= dk) return wfail(w, QP_ERR_ARG, "mask position out of range");
            P.push_back(positions[i]);
        }
    }
    std::sort(P.begin(), P.end());
    P.erase(std::unique(P.begin(), P.end()), P.end());
    if (P.empty() || P[0] != 0 || (dk >= 2 && (P.size() < 2 || P[1] != 1)))
        return wfail(w, QP_ERR_ARG, "mask must contain positions 0 and 1");
    const WParams keep = w->P;
    const qp_status s = wide_set_mask_params(w, P);
    if (s != QP_OK) {
        w->P = keep;
        return s;
    }
    w->mask = P;
    return QP_OK;
}

qp_status qp_wide_set_rho0(qp_wide *w, const double *re, const double *im) {
    if (!w) return QP_ERR_ARG;
    if (!re) return wfail(w, QP_ERR_ARG, "rho0 required");
    if (!w->have_eta) return wfail(w, QP_ERR_STATE, "qp_wide_set_eta must come before qp_wide_set_rho0");
    if (w->P.pp.npos < 0) return wfail(w, QP_ERR_STATE, "set a mask whose P' fits the 64-bit group key first");
    const int M = w->cfg.M, MM = M * M;
    std::vector<unsigned long long> lo, hi;
    std::vector<double2> amps, rho(MM);
    for (int a = 0; a < M; ++a)
        for (int b = 0; b < M; ++b) {
            const double x = re[a * M + b], y = im ? im[a * M + b] : 0.0;
            if (!std::isfinite(x) || !std::isfinite(y)) return wfail(w, QP_ERR_ARG, "rho0 must be finite");
            rho[a * M + b] = make_double2(x, y);
            if (x != 0.0 || y != 0.0) {
                lo.push_back((unsigned long long)(a | (b << 4)));
                hi.push_back(0ull);
                amps.push_back(make_double2(x, y));
            }
        }
    const size_t n = lo.size();
    std::vector<float2> af(n);
    for (size_t i = 0; i < n; ++i) af[i] = make_float2((float)amps[i].x, (float)amps[i].y);
    const size_t ab = w->P.c64 ? 8 : 16;
    QW_CUDA(w, cudaMemcpyAsync(w->P.klo[0], lo.data(), n * 8, cudaMemcpyHostToDevice, w->stream));
    QW_CUDA(w, cudaMemcpyAsync(w->P.khi[0], hi.data(), n * 8, cudaMemcpyHostToDevice, w->stream));
    QW_CUDA(w, cudaMemcpyAsync(w->P.amps[0], w->P.c64 ? (const void *)af.data() : (const void *)amps.data(), n * ab,
                               cudaMemcpyHostToDevice, w->stream));
    WState s{};
    s.n_cur = n;
    QW_CUDA(w, cudaMemcpyAsync(w->P.st, &s, sizeof(WState), cudaMemcpyHostToDevice, w->stream));
    QW_CUDA(w, cudaMemcpyAsync(w->P.rho_ring, rho.data(), MM * sizeof(double2), cudaMemcpyHostToDevice, w->stream));
    WRec r0{0, 0, 0, (long long)n, (long long)n};
    QW_CUDA(w, cudaMemcpyAsync(w->P.stats, &r0, sizeof(WRec), cudaMemcpyHostToDevice, w->stream));
    k_w_clear_table<<<std::max(1, w->nsm) * 4, 256, 0, w->stream>>>(w->P.slots, w->P.ttie,
                                                                    w->L.tcap);
    QW_CUDA(w, cudaGetLastError());
    QW_CUDA(w, cudaStreamSynchronize(w->stream));
    w->have_state = true;
    w->failed = false;
    return QP_OK;
}

qp_status qp_wide_step(qp_wide *w, int nsteps) {
    if (!w) return QP_ERR_ARG;
    if (nsteps < 0) return wfail(w, QP_ERR_ARG, "nsteps < 0");
    if (!w->have_state) return wfail(w, QP_ERR_STATE, "qp_wide_set_rho0 must come before qp_wide_step");
    if (w->failed) return wfail(w, QP_ERR_STATE, "context holds a device error; call qp_wide_set_rho0");
    if (nsteps == 0) return QP_OK;
    // the step count on the host decides merge or fill: read t once
    WState s;
    qp_status r = wide_read_state(w, &s);
    if (r != QP_OK) return r;
    unsigned long long t = s.t;
    for (int k = 0; k < nsteps; ++k, ++t) {
        const int merge = t + 1 >= (unsigned long long)w->cfg.dkmax ? 1 : 0;
        if (merge) {
            k_w_insert<<<w->nblk, kWThreads, 0, w->stream>>>(w->P);
            k_w_tie<<<w->nblk, kWThreads, 0, w->stream>>>(w->P);
        }
        if (w->P.c64) k_w_expand<true><<<w->xblk, kWThreads, w->xsmem, w->stream>>>(w->P, merge);
        else k_w_expand<false><<<w->xblk, kWThreads, w->xsmem, w->stream>>>(w->P, merge);
        k_w_finalize<<<1, 1024, 0, w->stream>>>(w->P, w->xblk, merge);
        QW_CUDA(w, cudaGetLastError());
    }
    return QP_OK;
}

qp_status qp_wide_current(qp_wide *w, int64_t *t, int64_t *n) {
    if (!w) return QP_ERR_ARG;
    if (!w->have_state) return wfail(w, QP_ERR_STATE, "no state");
    WState s;
    const qp_status r = wide_read_state(w, &s);
    if (t) *t = (int64_t)s.t;
    if (n) *n = (int64_t)s.n_cur;
    return r;
}

qp_status qp_wide_read_rho(qp_wide *w, int64_t t0, int count, double *re, double *im) {
    if (!w) return QP_ERR_ARG;
    if (!re || !im || count < 0) return wfail(w, QP_ERR_ARG, "bad output");
    if (!w->have_state) return wfail(w, QP_ERR_STATE, "no state");
    WState s;
    qp_status r = wide_read_state(w, &s);
    if (r != QP_OK) return r;
    const int MM = w->cfg.M * w->cfg.M;
    const int64_t R = w->P.rho_hist;
    if (t0 < 0 || t0 + count - 1 > (int64_t)s.t || (int64_t)s.t - t0 >= R) return wfail(w, QP_ERR_ARG, "t outside the kept history");
    std::vector<double2> buf((size_t)MM);
    for (int k = 0; k < count; ++k) {
        const int64_t t = t0 + k;
        QW_CUDA(w, cudaMemcpyAsync(buf.data(), w->P.rho_ring + (size_t)(t % R) * MM, MM * sizeof(double2),
                                   cudaMemcpyDeviceToHost, w->stream));
        QW_CUDA(w, cudaStreamSynchronize(w->stream));
        for (int i = 0; i < MM; ++i) {
            re[(size_t)k * MM + i] = buf[i].x;
            im[(size_t)k * MM + i] = buf[i].y;
        }
    }
    return QP_OK;
}

qp_status qp_wide_read_stats(qp_wide *w, int64_t t0, int count, qp_step_stats *out) {
    if (!w) return QP_ERR_ARG;
    if (!out || count < 0) return wfail(w, QP_ERR_ARG, "bad output");
    WState s;
    qp_status r = wide_read_state(w, &s);
    if (r != QP_OK) return r;
    const int64_t R = w->P.rho_hist;
    if (t0 < 0 || t0 + count - 1 > (int64_t)s.t || (int64_t)s.t - t0 >= R) return wfail(w, QP_ERR_ARG, "t outside the kept history");
    for (int k = 0; k < count; ++k) {
        WRec rec;
        QW_CUDA(w, cudaMemcpyAsync(&rec, w->P.stats + (size_t)((t0 + k) % R), sizeof(WRec), cudaMemcpyDeviceToHost,
                                   w->stream));
        QW_CUDA(w, cudaStreamSynchronize(w->stream));
        out[k].t = rec.t;
        out[k].groups = rec.groups;
        out[k].extended = rec.extended;
        out[k].kept = rec.kept;
        out[k].intermediate = rec.inter;
    }
    return QP_OK;
}

qp_status qp_wide_export_paths(qp_wide *w, uint64_t *keys, double *amps, int64_t cap, int64_t *n) {
    if (!w) return QP_ERR_ARG;
    if (!n || cap < 0 || (cap > 0 && (!keys || !amps))) return wfail(w, QP_ERR_ARG, "bad output");
    if (!w->have_state) return wfail(w, QP_ERR_STATE, "no state");
    WState s;
    qp_status r = wide_read_state(w, &s);
    if (r != QP_OK) return r;
    *n = (int64_t)s.n_cur;
    if ((int64_t)s.n_cur > cap) return wfail(w, QP_ERR_CAPACITY, "export buffer too small");
    const int buf = (int)(s.t & 1);
    const size_t cnt = s.n_cur;
    std::vector<unsigned long long> lo(cnt), hi(cnt);
    std::vector<float2> af(w->P.c64 ? cnt : 0);
    std::vector<double2> ad(w->P.c64 ? 0 : cnt);
    QW_CUDA(w, cudaMemcpyAsync(lo.data(), w->P.klo[buf], cnt * 8, cudaMemcpyDeviceToHost, w->stream));
    QW_CUDA(w, cudaMemcpyAsync(hi.data(), w->P.khi[buf], cnt * 8, cudaMemcpyDeviceToHost, w->stream));
    if (w->P.c64)
        QW_CUDA(w, cudaMemcpyAsync(af.data(), w->P.amps[buf], cnt * 8, cudaMemcpyDeviceToHost, w->stream));
    else
        QW_CUDA(w, cudaMemcpyAsync(ad.data(), w->P.amps[buf], cnt * 16, cudaMemcpyDeviceToHost, w->stream));
    QW_CUDA(w, cudaStreamSynchronize(w->stream));
    for (size_t i = 0; i < cnt; ++i) {
        keys[2 * i] = lo[i];
        keys[2 * i + 1] = hi[i];
        amps[2 * i] = w->P.c64 ? af[i].x : ad[i].x;
        amps[2 * i + 1] = w->P.c64 ? af[i].y : ad[i].y;
    }
    return QP_OK;
}

const char *qp_wide_last_error(const qp_wide *w) { return w ? w->err.c_str() : "null context"; }

}  // extern "C"
