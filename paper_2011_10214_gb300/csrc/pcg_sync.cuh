// Grid-wide synchronisation of the persistent PCG kernels (pcg_coop.cu,
// pcg_mg.cu): deterministic exchanges of block partials over a monotonic
// arrival counter, the fixed-point exchange of the FP32 inner loops, and a
// plain grid barrier.  Every wait is bounded (about a second at 2 GHz); a
// timeout sets ERR_BARRIER_TIMEOUT and the caller ends its solve.
#pragma once
#include "field_common.cuh"
#include "internal.h"

namespace pf {

struct ExchShared {
    double sh[4 * 32];
    double bc[4];
    int ok;
};

// grid exchange number e: publish this block's NV partials, wait for every
// block, return the grid totals (same in every block); false after a timeout.
// The barrier is one monotonic counter: each block adds 1 with release
// semantics and waits (acquire) until the count reaches the next multiple of
// the grid size -- no generation word, no reset, one atomic per block.
template <typename A, int NV, typename Args>
static __device__ __forceinline__ bool exchange(const Args& a, int& e, A (&v)[NV], A (&tot)[NV], ExchShared& xs) {
    A* sh = (A*)xs.sh;
    block_sum_t<A, NV>(v, sh);                // ends with __syncthreads: the block's z stores are issued
    const unsigned G = gridDim.x;
    A* val = (A*)a.val + (size_t)(e & 1) * 4 * G;
    const bool first_of_launch = e == 0;
    ++e;
    if (threadIdx.x == 0) {
#pragma unroll
        for (int q = 0; q < NV; ++q) __stcg(val + (size_t)q * G + blockIdx.x, v[q]);
        const unsigned long long t = atom_add_release(a.arrivals, 1ull);
        // (a test can make the launch's first exchange wait for arrivals that
        // never come, to see the bounded wait give up and report)
        const unsigned long long target = (t / G + 1) * G + (first_of_launch ? (unsigned long long)*a.hold : 0ull);
        int ok = 1;
        if (ld_acquire(a.arrivals) < target) {
            const long long c0 = clock64();
            while (ld_acquire(a.arrivals) < target)
                if (clock64() - c0 > (1ll << 31)) { ok = 0; atomicOr(a.err, ERR_BARRIER_TIMEOUT); break; }
        }
        xs.ok = ok;
    }
    __syncthreads();
    if (!xs.ok) return false;
    A* bc = (A*)xs.bc;
    if constexpr (std::is_same<A, double>::value) {   // (a value per warp: the adds of FP64)
        const int q = threadIdx.x >> 5, lane = threadIdx.x & 31;
        if (q < NV) {
            double s = 0.0;
            for (unsigned g0 = 0; g0 < G; g0 += 160) {
                double p[5];
#pragma unroll
                for (int k = 0; k < 5; ++k) {
                    const unsigned g = g0 + 32 * k + lane;
                    p[k] = g < G ? __ldcg(val + (size_t)q * G + g) : 0.0;
                }
                s += ((p[0] + p[1]) + (p[2] + p[3])) + p[4];
            }
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
            if (lane == 0) bc[q] = s;
        }
    } else {
        A s[NV];
#pragma unroll
        for (int q = 0; q < NV; ++q) s[q] = threadIdx.x < G ? __ldcg(val + (size_t)q * G + threadIdx.x) : (A)0;
        block_sum_t<A, NV>(s, sh);
        if (threadIdx.x == 0)
#pragma unroll
            for (int q = 0; q < NV; ++q) bc[q] = s[q];
    }
    __syncthreads();
#pragma unroll
    for (int q = 0; q < NV; ++q) tot[q] = bc[q];
    return true;
}

// ---- fixed-point exchange (FP32 inner loop of the register-resident kernel) ----
//
// The arrival and the partial travel in one fire-and-forget atomic: a block
// adds to one 64-bit word per value
//     (rint(v 2^k) << 2W) + (fits ? 1 : 1 + 2^W)
// -- bits 0..W-1 count arrivals, bits W..2W-1 blocks whose scaled partial did
// not fit, bits 2W..63 the two's-complement sum.  W = 8 (at most 255 blocks):
// partials below 2^39, a 48-bit sum, the scale 2^k puts the value's previous
// total near 2^32; W = 9 (at most 511 blocks): partials below 2^36, a 46-bit
// sum, previous total near 2^29.  No field carries into the next within one
// exchange.  A block polls the word until its growth since the previous use
// shows every arrival; the growth then holds the integer total, each partial
// exact to 2^-32 (2^-29) of the previous total.  Integer sums do not depend on the
// arrival order: results stay deterministic run to run.  A word is reused only
// after the other exchange kind (a full barrier) has passed, so its value is
// stable from the last arrival until every block has read it.  If a partial
// did not fit, or the total kept fewer than 2^26 (2^23) units (the value fell
// far below its previous total), every block sees it and redoes the values
// with the partial exchange above.
constexpr int FX_LINE = 16;                  // words per 128-byte line
template <int W>
struct FxLayout {
    static_assert(W == 8 || W == 9, "layouts for up to 255 or 511 blocks");
    static constexpr int SUM = 2 * W;                                        // sum field shift
    static constexpr unsigned long long MASK = (1ull << W) - 1;
    static constexpr float FIT = W == 8 ? 549755813888.0f : 68719476736.0f;   // 2^39, 2^36
    static constexpr int SCALE = W == 8 ? 32 : 29;
    static constexpr long long MIN = W == 8 ? (1ll << 26) : (1ll << 23);
};

// ref: the previous totals (positive, normal); prev: this lane's word value
// after its last use (lanes 0..NV-1 of warp 0).  Returns 1 with the totals in
// tot, -1 if the values must be redone, 0 after a timeout.
template <int NV, bool REL, int W, typename Args>
static __device__ __forceinline__ int exchange_fx(const Args& a, unsigned long long* words, unsigned long long& prev,
                                                  const float (&ref)[NV], float (&v)[NV], float (&tot)[NV],
                                                  ExchShared& xs) {
    block_sum_t<float, NV>(v, (float*)xs.sh);   // totals in thread 0; ends with __syncthreads
    float* bc = (float*)xs.bc;
    if (threadIdx.x < 32) {
        const int lane = threadIdx.x;
        const bool act = lane < NV;
        float mine = 0.0f, rf = ref[0];
#pragma unroll
        for (int q = 0; q < NV; ++q) {      // lane q takes value q (the block total sits in thread 0)
            const float t = __shfl_sync(0xffffffffu, v[q], 0);
            if (lane == q) { mine = t; rf = ref[q]; }
        }
        using FL = FxLayout<W>;
        const int k = FL::SCALE - ilogbf(rf);
        const float sc = ldexpf(mine, k);
        const bool fits = fabsf(sc) < FL::FIT;
        const long long fx = fits ? __float2ll_rn(sc) : 0ll;
        unsigned long long* w = words + lane * FX_LINE;
        if (act) {
            const unsigned long long add = ((unsigned long long)fx << FL::SUM) + (fits ? 1ull : 1ull + (1ull << W));
            if (REL) red_add_release(w, add);
            else red_add_relaxed(w, add);
        }
        const unsigned long long G = gridDim.x;
        unsigned long long d = 0;
        bool done = !act, timeout = false;
        const long long c0 = clock64();
        for (;;) {
            if (!done) {
                d = ld_acquire(w) - prev;
                done = (d & FL::MASK) == G;
            }
            if (__all_sync(0xffffffffu, done)) break;
            if (__any_sync(0xffffffffu, clock64() - c0 > (1ll << 31))) { timeout = true; break; }
        }
        bool good = true;
        if (act && !timeout) {
            prev += d;
            const long long val = (long long)d >> FL::SUM;
            good = ((d >> W) & FL::MASK) == 0 && (val >= FL::MIN || val <= -FL::MIN);
            bc[lane] = ldexpf((float)val, -k);
        }
        const bool all_good = __all_sync(0xffffffffu, good);
        if (lane == 0) {
            if (timeout) atomicOr(a.err, ERR_BARRIER_TIMEOUT);
            xs.ok = timeout ? 0 : (all_good ? 1 : 2);
        }
    }
    __syncthreads();
    // (the next exchange rewrites bc and ok only after its block sum's barrier)
    const int ok = xs.ok;
    if (ok == 1) {
#pragma unroll
        for (int q = 0; q < NV; ++q) tot[q] = bc[q];
    }
    return ok == 1 ? 1 : (ok == 2 ? -1 : 0);
}

// an FP32 exchange: fixed-point when the previous totals give a scale, else
// (or when the fixed-point totals cannot be trusted) the partial exchange
template <int NV, bool REL, int W, typename Args>
static __device__ __forceinline__ bool exchange_f32(const Args& a, int& e, unsigned long long* words,
                                                    unsigned long long& prev, const float (&ref)[NV], bool use_fx,
                                                    float (&v)[NV], float (&tot)[NV], ExchShared& xs) {
    if (use_fx) {
        float vc[NV];
#pragma unroll
        for (int q = 0; q < NV; ++q) vc[q] = v[q];
        const int rc = exchange_fx<NV, REL, W>(a, words, prev, ref, vc, tot, xs);
        if (rc == 1) return true;
        if (rc == 0) return false;
    }
    return exchange<float, NV>(a, e, v, tot, xs);
}

// ---- the same for FP64 values -------------------------------------------------
//
// An FP64 add takes a scheduler 67 cycles and the grid's partials a round trip
// of their own, so an exchange of FP64 sums (block sums twice, partials through
// memory) took 4.6 us of a 10 us iteration.  Here a thread's value becomes an
// integer in units of 2^-72 of its previous total's power of two, cut into three
// signed pieces of 26 bits: warps add the pieces with one integer reduction
// each, a block adds each to a 64-bit word of its own (layout W = 8: arrivals,
// misfits, a 48-bit sum, which 255 blocks of 2^35 cannot fill), and every block
// puts the three totals together.  A value is rounded once, to 2^-72 of the
// previous total, and everything after that is exact: less error than the FP64
// sums, and the same in any order.  A value above 32 previous totals, or a total
// below 1/128 of it, is redone with the partial exchange.
// 2.8 us an exchange at 16^3 nodes; with the closed-form rows, an iteration went
// from 17 to 8 us there and from 22 to 11 us at 40^3.
template <int NV, bool REL, typename Args, typename F>
static __device__ __forceinline__ int exchange_fx64(const Args& a, unsigned long long* words, unsigned long long& prev,
                                                    const double (&ref)[NV], const double (&v)[NV], double (&tot)[NV],
                                                    F ratio, double& quot, ExchShared& xs) {
    using FL = FxLayout<8>;
    constexpr int NP = 3 * NV;
    constexpr unsigned PIECE = (1u << 26) - 1;
    int* part = (int*)xs.sh;                       // [NP][warps], then the warps' misfits
    static_assert(sizeof(xs.sh) >= sizeof(int) * 16 * (NP + 1), "at most 16 warps");
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, nw = blockDim.x >> 5;
    int er[NV];
    bool fits = true;
#pragma unroll
    for (int q = 0; q < NV; ++q) {
        er[q] = (int)((__double_as_longlong(ref[q]) >> 52) & 0x7ff);
        const long long bits = __double_as_longlong(v[q]);
        const int ex = (int)((bits >> 52) & 0x7ff), up = ex - er[q] + 20;
        unsigned long long m = ex ? ((unsigned long long)bits & ((1ull << 52) - 1)) | (1ull << 52) : 0ull, hi = 0;
        fits = fits && up <= 24;                   // (infinities and NaN do not fit either)
        if (up > 0) {
            hi = m >> (64 - min(up, 24));
            m <<= min(up, 24);
        } else {
            const int s = min(-up, 63);
            m = (m + ((1ull << s) >> 1)) >> s;
        }
        int piece[3] = {(int)((unsigned)m & PIECE), (int)((unsigned)(m >> 26) & PIECE),
                        (int)((unsigned)(m >> 52) | (unsigned)(hi << 12))};
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            const int sum = __reduce_add_sync(0xffffffffu, bits < 0 ? -piece[c] : piece[c]);
            if (lane == 0) part[(3 * q + c) * 16 + wid] = sum;
        }
    }
    fits = __all_sync(0xffffffffu, fits);
    if (lane == 0) part[NP * 16 + wid] = fits ? 0 : 1;
    __syncthreads();                               // (the block's z stores are issued)
    if (wid == 0) {
        const bool act = lane < NP;
        const bool bad = __any_sync(0xffffffffu, lane < nw && part[NP * 16 + (lane & 15)] != 0);
        long long sum = 0;
        if (act && !bad)
            for (int w = 0; w < nw; ++w) sum += part[lane * 16 + w];
        unsigned long long* w = words + (act ? lane : 0) * FX_LINE;
        if (act) {
            const unsigned long long add = ((unsigned long long)sum << FL::SUM) + (bad ? 1ull + (1ull << 8) : 1ull);
            if (REL) red_add_release(w, add);
            else red_add_relaxed(w, add);
        }
        const unsigned long long G = gridDim.x;
        unsigned long long d = 0;
        bool done = !act, timeout = false;
        const long long c0 = clock64();
        for (;;) {
            if (!done) {
                d = ld_acquire(w) - prev;
                done = (d & FL::MASK) == G;
            }
            if (__all_sync(0xffffffffu, done)) break;
            if (__any_sync(0xffffffffu, clock64() - c0 > (1ll << 31))) { timeout = true; break; }
        }
        if (act && !timeout) prev += d;
        bool good = !__any_sync(0xffffffffu, act && ((d >> 8) & FL::MASK) != 0);
        const long long val = (long long)d >> FL::SUM;
        double t[NV];
#pragma unroll
        for (int q = 0; q < NV; ++q) {
            const long long p0 = __shfl_sync(0xffffffffu, val, 3 * q), p1 = __shfl_sync(0xffffffffu, val, 3 * q + 1),
                            p2 = __shfl_sync(0xffffffffu, val, 3 * q + 2);
            const __int128 all = ((__int128)p2 << 52) + ((__int128)p1 << 26) + p0;
            const unsigned __int128 mag = all < 0 ? -(unsigned __int128)all : (unsigned __int128)all;
            const unsigned long long mh = (unsigned long long)(mag >> 64);
            const int top = mh ? 127 - __clzll((long long)mh) : 63 - __clzll((long long)(unsigned long long)mag);
            if (top < 66) good = false;
            // round to 53 bits; a carry out of the mantissa raises the exponent
            const int s = top > 53 ? top - 52 : 1;
            const unsigned long long m53 = (unsigned long long)((mag + ((unsigned __int128)1 << (s - 1))) >> s);
            const unsigned long long out = ((unsigned long long)(top + er[q] - 73) << 52) + m53;
            t[q] = __longlong_as_double((long long)(out | (all < 0 ? 1ull << 63 : 0ull)));
        }
        if (lane == 0) {
            if (timeout) atomicOr(a.err, ERR_BARRIER_TIMEOUT);
            xs.ok = timeout ? 0 : good ? 1 : 2;
#pragma unroll
            for (int q = 0; q < NV; ++q) xs.bc[q] = t[q];
            xs.bc[3] = timeout || !good ? 0.0 : ratio(t);
        }
    }
    __syncthreads();
    const int ok = xs.ok;
    if (ok == 1) {
#pragma unroll
        for (int q = 0; q < NV; ++q) tot[q] = xs.bc[q];
        quot = xs.bc[3];
    }
    return ok == 1 ? 1 : (ok == 2 ? -1 : 0);
}

// an FP64 exchange with a quotient of its totals: fixed-point when the previous
// totals give a scale, else the partial exchange
template <int NV, bool REL, typename Args, typename F>
static __device__ __forceinline__ bool exchange_f64(const Args& a, int& e, unsigned long long* words,
                                                    unsigned long long& prev, const double (&ref)[NV], double (&v)[NV],
                                                    double (&tot)[NV], F ratio, double& quot, ExchShared& xs) {
    bool use = true;
#pragma unroll
    for (int q = 0; q < NV; ++q) {
        // positive, 2^-663 to 2^664 (by its bits: every warp would compare in FP64)
        const unsigned hi = (unsigned)__double2hiint(ref[q]) >> 20;
        use = use && hi > 360u && hi < 1687u;
    }
    if (use) {
        const int rc = exchange_fx64<NV, REL>(a, words, prev, ref, v, tot, ratio, quot, xs);
        if (rc >= 0) return rc == 1;
    }
    const bool ok = exchange<double, NV>(a, e, v, tot, xs);
    quot = ok ? ratio(tot) : 0.0;
    return ok;
}

// a previous total usable as the fixed-point scale
static __device__ __forceinline__ bool fx_ref_ok(float r) { return r > 1e-30f && r < 1e30f; }


// grid barrier number e (shares the arrival counter and the bounded wait of
// the exchanges, carries no values); false after a timeout.  The block's
// stores before the call are visible to every block after it returns.
template <typename Args>
static __device__ __forceinline__ bool grid_barrier(const Args& a, int& e, ExchShared& xs) {
    __syncthreads();
    const unsigned G = gridDim.x;
    const bool first_of_launch = e == 0;
    ++e;
    if (threadIdx.x == 0) {
        const unsigned long long t = atom_add_release(a.arrivals, 1ull);
        const unsigned long long target = (t / G + 1) * G + (first_of_launch ? (unsigned long long)*a.hold : 0ull);
        int ok = 1;
        if (ld_acquire(a.arrivals) < target) {
            const long long c0 = clock64();
            while (ld_acquire(a.arrivals) < target)
                if (clock64() - c0 > (1ll << 31)) { ok = 0; atomicOr(a.err, ERR_BARRIER_TIMEOUT); break; }
        }
        xs.ok = ok;
    }
    __syncthreads();
    return xs.ok != 0;
}

}  // namespace pf
