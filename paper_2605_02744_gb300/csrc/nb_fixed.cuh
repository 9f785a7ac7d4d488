// Exact, order-independent accumulation of floating-point partial sums in
// two-word fixed point, for sums that many CTAs add to at once.
//
// A call fixes one exponent F for every accumulator.  A partial sum v (FP32
// or FP64) becomes the integer X = v 2^F rounded half away from zero (in
// integer arithmetic on the bits of v), split as X = hi 2^40 + lo
// with 0 <= lo < 2^40; hi goes into one 64-bit word and lo into another with
// integer atomic adds.  Integer addition is associative, so the words end the
// same whatever order the adds arrive in: results are bitwise reproducible,
// and the only rounding is the one of each partial to the grid 2^-F.  F is
// chosen from an a-priori bound Bd on every partial and on every total
// (|X| < 2^100), so the words cannot overflow: |hi| < 2^60 per add, and lo
// has 24 bits of headroom (2^24 adds per accumulator).
#pragma once

#include <cuda_runtime.h>
#include <math.h>
#include <stdint.h>
#include <string.h>

#include "nb_internal.h"

namespace nb {
namespace fx {

constexpr int kLoBits = 40;
constexpr int kMagBits = 100;  // |X| < 2^100

// Exponent for totals bounded by `bound` (>= 0): bound 2^F < 2^100.
__host__ __device__ inline int exponent_for(double bound) {
    if (!(bound > 0.0)) return 0;          // all partials are zero
    if (!isfinite(bound)) return -900;     // the FP32 / FP64 sums overflow first
    int e = 0;
    frexp(bound, &e);                      // bound < 2^e
    int F = kMagBits - e;
    return F < -900 ? -900 : (F > 900 ? 900 : F);
}

// The two words' increments (hi, lo) of an FP64 partial v, in integer
// arithmetic on its bits (no FP64 operations, which are slow on this part):
// with v = m 2^(k - 52), m the 53-bit significand, X = m 2^(k - 52 + F) is m
// shifted left (exact) or right (rounded half away from zero), split as
// |X| = H 2^40 + L and negated in two's complement for v < 0.  false (no
// increments) if v is not finite or |X| >= 2^100.  The same source runs on
// the host, where nb_check_fp_conversions checks it.
__host__ __device__ inline bool split_f64(double v, int F, unsigned long long &hi,
                                          unsigned long long &lo) {
    unsigned long long b;
    memcpy(&b, &v, 8);
    const int be = (int)((b >> 52) & 0x7ffu);
    hi = lo = 0;
    if (be == 0x7ff) return false;  // inf or NaN
    unsigned long long m = b & 0xfffffffffffffull;
    if (be) m |= 1ull << 52;
    if (!m) return true;  // +-0
    const int s = (be ? be : 1) - 1075 + F;  // X = m 2^s
    unsigned __int128 X;
    if (s >= 0) {
        if (s > kMagBits - 53) return false;  // beyond the bound
        X = (unsigned __int128)m << s;
    } else {
        if (s < -54) return true;  // below half a grid step
        X = ((unsigned __int128)m + ((unsigned __int128)1 << (-s - 1))) >> (-s);
    }
    if (X >> kMagBits) return false;
    const unsigned long long H = (unsigned long long)(X >> kLoBits);
    const unsigned long long L = (unsigned long long)X & ((1ull << kLoBits) - 1);
    if (b >> 63) {  // two's complement of H 2^40 + L
        hi = L ? ~H : (0ull - H);
        lo = L ? (1ull << kLoBits) - L : 0ull;
    } else {
        hi = H;
        lo = L;
    }
    return true;
}

// Adds v to accumulator (word_hi, word_lo); false (nothing added) if v is
// not finite or outside the bound.
__device__ __forceinline__ bool add(unsigned long long *word_hi, unsigned long long *word_lo,
                                    double v, int F) {
    unsigned long long hi, lo;
    if (!split_f64(v, F, hi, lo)) return false;
    if (hi) atomicAdd(word_hi, hi);
    if (lo) atomicAdd(word_lo, lo);
    return true;
}

// add() for an FP32 partial, in integer arithmetic on its bits (no FP64
// operations, which are slow on this part): with v = m 2^(k - 23), m the
// 24-bit significand, X = m 2^(k - 23 + F) is m shifted left (exact) or
// right (rounded half away from zero; the result is the same for any
// arrival order either way).
__device__ __forceinline__ bool add_f32(unsigned long long *word_hi,
                                        unsigned long long *word_lo, float v, int F) {
    const uint32_t b = __float_as_uint(v);
    const int be = (int)((b >> 23) & 0xffu);
    if (be == 0xff) return false;  // inf or NaN
    uint32_t m = b & 0x7fffffu;
    if (be) m |= 0x800000u;
    if (!m) return true;  // +-0
    const int s = (be ? be : 1) - 150 + F;  // X = m 2^s
    unsigned long long H, L;                // |X| = H 2^40 + L
    if (s >= 0) {
        if (s > kMagBits - 24) return false;  // beyond the bound
        if (s >= kLoBits) {
            H = (unsigned long long)m << (s - kLoBits);
            L = 0;
        } else {
            const unsigned long long X = (unsigned long long)m << s;  // < 2^64
            H = X >> kLoBits;
            L = X & ((1ull << kLoBits) - 1);
        }
    } else {
        if (s < -25) return true;  // below half a grid step
        H = 0;
        L = ((unsigned long long)m + (1ull << (-s - 1))) >> (-s);
    }
    unsigned long long hi, lo;
    if (b >> 31) {  // two's complement of H 2^40 + L
        hi = L ? ~H : (0ull - H);
        lo = L ? (1ull << kLoBits) - L : 0ull;
    } else {
        hi = H;
        lo = L;
    }
    if (hi) atomicAdd(word_hi, hi);
    if (lo) atomicAdd(word_lo, lo);
    return true;
}

// A magnitude m (nonzero) as sign 2^53-significand double m 2^(-shift),
// rounded to nearest even in integer arithmetic (ldexp and the FP64
// conversions are slow on this part); results below the smallest normal
// double go through ldexp.
__host__ __device__ inline double scaled(unsigned __int128 m, int shift, bool neg) {
    const unsigned long long mh = (unsigned long long)(m >> 64), ml = (unsigned long long)m;
#ifdef __CUDA_ARCH__
    const int lz = mh ? __clzll((long long)mh) : 64 + __clzll((long long)ml);
#else
    const int lz = mh ? __builtin_clzll(mh) : 64 + __builtin_clzll(ml);
#endif
    const int top = 127 - lz;  // bit of the leading one
    unsigned long long K;      // 53 significant bits
    if (top <= 52) {
        K = ml << (52 - top);
    } else {
        const int sh = top - 52;
        K = (unsigned long long)(m >> sh);
        const unsigned __int128 rest = m & (((unsigned __int128)1 << sh) - 1);
        const unsigned __int128 half = (unsigned __int128)1 << (sh - 1);
        if (rest > half || (rest == half && (K & 1ull))) ++K;  // 2^53: the exponent moves up
    }
    const int e = top + 1023 - shift;
    double d;
    if (e >= 1 && e < 2046) {
        const unsigned long long b = ((unsigned long long)(e - 1) << 52) + K;
        memcpy(&d, &b, 8);
    } else {
        d = ldexp((double)K, top - 52 - shift);
    }
    return neg ? -d : d;
}

// The accumulated value: (signed) hi 2^40 + lo, exactly as a 128-bit
// integer, then rounded once to double and scaled by 2^-F.
__host__ __device__ inline double value(unsigned long long word_hi, unsigned long long word_lo,
                                        int F) {
    const __int128 t = ((__int128)(long long)word_hi) * ((__int128)1 << kLoBits) +
                       (__int128)word_lo;
    if (!t) return 0.0;
    return scaled(t < 0 ? (unsigned __int128)(-t) : (unsigned __int128)t, F, t < 0);
}

// ------------------------------------------------------------- four limbs
// The same with four signed limbs of 44 bits, X = sum L_q 2^(44 q), for the
// warp-granular kernels: their VJP and jerk bounds grow with eps^-3, and 100
// bits below them would be coarser than the FP32 pair terms once eps is below
// ~1e-6 of the system size; 174 bits are not before ~1e-11 of it, and from there
// the grid of the FP32-pair kernels no longer follows eps
// (wsym::length_exponent).  A 24-bit significand touches one limb, or
// two where it straddles a boundary, whatever its sign.  19 bits of headroom:
// 2^19 adds per accumulator.
constexpr int kLimbs = 4, kLimbBits = 44;
constexpr int kLimbMagBits = kLimbs * kLimbBits - 2;  // |X| < 2^174

// The exponent of a bound that is not finite: no grid, every total a NaN.
constexpr int kNoGrid = -100000;
// A partial that is not finite, or beyond the bound, poisons its accumulator:
// atomicMax of the top limb with this value, 2^18 times what sums reach there,
// and the total reads as a NaN.
constexpr long long kPoison = 1ll << 62;

__host__ __device__ inline int limb_exponent_for(double bound) {
    if (!isfinite(bound)) return kNoGrid;
    if (!(bound > 0.0)) return 0;
    int e = 0;
    frexp(bound, &e);  // bound < 2^e
    const int F = kLimbMagBits - e;
    return F < -900 ? -900 : (F > 900 ? 900 : F);
}

// The same from an exponent e with bound < 2^e (kNoBound: not finite).
constexpr int kNoBound = 4096;
__host__ __device__ inline int limb_exponent(int e) {
    if (e >= kNoBound / 2) return kNoGrid;
    const int F = kLimbMagBits - e;
    return F < -900 ? -900 : (F > 900 ? 900 : F);
}

// v 2^F rounded half away from zero: limb q gains lo, limb q + 1 hi (both with
// v's sign; zeros need no add).  false (no increments) if v is not finite or
// beyond the limbs.
__host__ __device__ inline bool split_limbs(float v, int F, int &q, long long &lo, long long &hi) {
    uint32_t b;
    memcpy(&b, &v, 4);
    const int be = (int)((b >> 23) & 0xffu);
    q = 0;
    lo = hi = 0;
    if (be == 0xff) return false;  // inf or NaN
    uint32_t m = b & 0x7fffffu;
    if (be) m |= 0x800000u;
    if (!m) return true;  // +-0
    int s = (be ? be : 1) - 150 + F;  // X = m 2^s
    unsigned long long M = m;
    if (s < 0) {
        if (s < -25) return true;  // below half a grid step
        M = (M + (1ull << (-s - 1))) >> (-s);
        s = 0;
    }
    q = s / kLimbBits;
    const int r = s - q * kLimbBits;
    const unsigned long long l = (M << r) & ((1ull << kLimbBits) - 1), h = M >> (kLimbBits - r);
    if (q >= kLimbs || (q == kLimbs - 1 && h)) {
        q = 0;
        return false;
    }
    lo = (b >> 31) ? -(long long)l : (long long)l;
    hi = (b >> 31) ? -(long long)h : (long long)h;
    return true;
}

// The same for an FP64 value: limbs q, q + 1, q + 2 gain t[0..2].
__host__ __device__ inline bool split_limbs(double v, int F, int &q, long long (&t)[3]) {
    unsigned long long b;
    memcpy(&b, &v, 8);
    const int be = (int)((b >> 52) & 0x7ffu);
    q = 0;
    t[0] = t[1] = t[2] = 0;
    if (be == 0x7ff) return false;  // inf or NaN
    unsigned long long m = b & 0xfffffffffffffull;
    if (be) m |= 1ull << 52;
    if (!m) return true;  // +-0
    int s = (be ? be : 1) - 1075 + F;  // X = m 2^s
    if (s < 0) {
        if (s < -54) return true;  // below half a grid step
        m = (m + (1ull << (-s - 1))) >> (-s);
        s = 0;
    }
    const unsigned long long mask = (1ull << kLimbBits) - 1;
    q = s / kLimbBits;
    const int r = s - q * kLimbBits;
    const unsigned __int128 X = (unsigned __int128)m << r;  // < 2^97
    const unsigned long long l[3] = {(unsigned long long)X & mask,
                                     (unsigned long long)(X >> kLimbBits) & mask,
                                     (unsigned long long)(X >> (2 * kLimbBits))};
    if (q >= kLimbs || (q >= kLimbs - 1 && l[1]) || (q >= kLimbs - 2 && l[2])) {
        q = 0;
        return false;
    }
#pragma unroll
    for (int k = 0; k < 3; ++k) t[k] = (b >> 63) ? -(long long)l[k] : (long long)l[k];
    return true;
}

// The accumulated value of the limbs, rounded once to double; a NaN for a
// poisoned accumulator or without a grid.
__host__ __device__ inline double limb_value(const long long (&w)[kLimbs], int F) {
    if (F == kNoGrid || w[kLimbs - 1] >= kPoison / 2) {
        const unsigned long long nan_bits = 0x7ff8000000000000ull;
        double d;
        memcpy(&d, &nan_bits, 8);
        return d;
    }
    long long t[kLimbs];
    long long c = 0;  // carries: every limb but the top one into [0, 2^44)
#pragma unroll
    for (int k = 0; k < kLimbs; ++k) {
        t[k] = w[k] + c;
        if (k + 1 < kLimbs) {
            c = t[k] >> kLimbBits;
            t[k] -= c * (1ll << kLimbBits);
        }
    }
    const bool neg = t[kLimbs - 1] < 0;
    if (neg) {  // the magnitude's limbs
        c = 0;
#pragma unroll
        for (int k = 0; k < kLimbs; ++k) {
            t[k] = c - t[k];
            if (k + 1 < kLimbs) {
                c = t[k] >> kLimbBits;
                t[k] -= c * (1ll << kLimbBits);
            }
        }
    }
    int shift = F;
    if (t[3] == 0) {  // the leading three limbs that hold anything
        t[3] = t[2];
        t[2] = t[1];
        t[1] = t[0];
        t[0] = 0;
        shift += kLimbBits;
    }
    if (t[3] == 0) {
        t[3] = t[2];
        t[2] = t[1];
        t[1] = 0;
        shift += kLimbBits;
    }
    if (t[3] == 0) {
        t[3] = t[2];
        t[2] = 0;
        shift += kLimbBits;
    }
    // t3 2^132 + t2 2^88 + t1 2^44 + t0 with t3 != 0 unless all are zero: 128
    // bits from 2^72 up (t3 < 2^63, so t3 2^60 fits), the rest as a sticky bit
    // (they only decide ties)
    const bool sticky = (t[1] & ((1ll << 28) - 1)) | t[0];
    const unsigned __int128 m = ((unsigned __int128)t[3] << 60) |
                                ((unsigned __int128)t[2] << 16) | ((unsigned __int128)t[1] >> 28) |
                                (sticky ? 1 : 0);
    if (!m) return 0.0;
    return scaled(m, shift - 72, neg);
}

}  // namespace fx
}  // namespace nb
