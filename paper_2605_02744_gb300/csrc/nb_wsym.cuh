// Warp-granular symmetric-pair evaluation of one system: the engine shared by
// the force (nb_wsym.cu), the VJP (nb_vjp.cu) and the acceleration + jerk
// (nb_jerk.cu) when every pair takes the same displacement form.
//
// Each unordered pair is evaluated once for both particles, as in nb_sym.cu.
// A warp keeps one block of i-slots in registers, four or eight per lane; the
// items are the block pairs (I, J >= I), row-major; an item is a few j-sets
// of 32 or 64 slots, a j-set 32 rotation steps: at step s lane l holds j-slot
// (l + s) mod 32 (of both halves of a 64-slot set), and after it everything a
// j-particle carries, its own sums included, moves one lane down.  Either an
// i-slot is broadcast as (x, x) against two j in the .x / .y halves, or two
// i-slots (IPAIR) against one broadcast j: every FP32 operation is packed.
//
// The step is the unit of work.  All steps of all items form one line that is
// cut into equal contiguous ranges, one per warp: a range may start or end in
// the middle of a rotation, because a lane can load the j-slot of any step
// directly and its sums can be added to whatever slot they have reached.  So
// every warp of the GPU gets the same number of pairs to within four steps at
// any N -- row blocks of 2048 slots and units of 2 x 64 j-slots left a
// 16384-particle evaluation with 3.8 units per SM, i.e. 5 % idle, and smaller
// ones with a handful of busy SMs -- and no warp waits for another inside the
// loop.  (The items on the diagonal do the i-side of all ordered pairs of
// their block: 60 to 75 % of the others' cost a step; they are 2 / nb of the
// steps.)
//
// Sums.  The terms of one rotation step for a j-particle go into fresh
// registers, then with one add into its travelling sum; a j-set's travelling
// sums (at most 256 terms) go into the particle's fixed-point totals
// (nb_fixed.cuh, four limbs: integer atomics, exact, so results do not depend on the
// order in which warps arrive).  The i-side register sums are folded every 4
// j-sets (128 terms per stream) into a total of the policy's own kind (Total
// below) in shared memory, and at the end of the
// warp's segment of a row into the same totals.  The warps of a CTA own
// consecutive ranges, so their last segments mostly belong to one row: these
// are added up in the same form across the CTA, in warp order,
// before the atomics.
//
// What bounds it: in part the register file.  A packed FMA with three distinct
// operands reads six registers and issues at 64 % of the FP32 peak (two
// distinct: 95 %; measured on chains of independent operations), and 6 of a
// force pair's 16, 17 of a jerk pair's 39 operations are of that kind, so that
// 80 to 83 % of the peak is the ceiling of the mix: 88 us for the pairs of 16384
// particles (hi/lo), which take about 117.  Of the rest the ends are a part (each
// warp's first loads, a row's end, the launch); the pipe is
// busy 69 % of the time within the kernel (ncu, 16384 particles)
// whatever the number of warps, the order of the operations in the source or
// the unrolling, and what else keeps it from 80 % is not known.  GB300, 16384
// particles, one evaluation with its pack and fold: F64ACC forces 194 -> 141
// us, acceleration + jerk 945 -> 232 us, VJP 332 -> 198 us against the direct
// kernels.
#pragma once

#include <cuda_runtime.h>
#include <math.h>
#include <stdint.h>

#include <algorithm>
#include <type_traits>

#include "nb_device.cuh"
#include "nb_fixed.cuh"
#include "nb_internal.h"

namespace nb {
namespace wsym {

using dev::add2;
using dev::f2;
using dev::fma2;
using dev::mul2;
using dev::rsqrt_approx;

constexpr int GR = 4;              // rotation steps per scheduling unit
constexpr int FLUSH = 4;           // j-sets per i-side flush (128 terms per stream)
constexpr int kMaxGroups = 3;

struct Params {
    const float *soa;    // [7 or 10][Np]: x.hi y.hi z.hi m x.lo y.lo z.lo (vx vy vz)
    const float *csoa;   // [4][Np]: cx cy cz pbar (VJP)
    int64_t Np;
    int64_t N;
    int64_t nb;          // blocks
    int64_t per_warp, extra;  // scheduling units per warp; the first `extra` warps take one more
    float eps;
    bool keep;           // KAHAN: compensated i-side sums; FP32: plain ones
    unsigned long long *fx;  // [components][4 limbs][Np] fixed-point totals
    int *fxe;                // [kMaxGroups] the call's exponents (written here)
    const unsigned *mx;      // maxima of the inputs (float bits), see MaxWord
    int sexp[5];             // exponents of the factors of the a-priori bounds (set_scale), see
                             // each physics' bound()
    void set_scale(int k, double v) { frexp(v, &sexp[k]); }  // v < 2^sexp[k]
    uint32_t *status;
};

// Words of `mx`: the largest |m|, |v|, |x| and |c| component and |pbar| of the
// packed inputs,
// as float bits rounded up (non-negative floats order like their bits).
enum MaxWord { kMaxM = 0, kMaxV = 1, kMaxX = 2, kMaxC = 3, kMaxP = 4 };

// Powers of two that bring the packed inputs to order one where they are
// loaded: lengths, masses, cotangents.  r^-3 leaves the range of FP32 at
// distances of 4e12 (metres, say), and products of masses and cotangents
// sooner; powers of two change no rounding, and the fold's exponents undo them.
struct Scales {
    int x, m, c;
};
// The exponent of the unit of length, from those of max|x| and eps (v < 2^e):
// max|x| itself, unless eps is so much smaller that eps^-3 would leave FP32
// (one escaper at 10^6 with eps = 1e-8: the unit follows eps, whose inverse
// cube stays below 2^111, with room for a jerk's velocity) or larger (x^-3 is
// then eps^-3, and the accelerations, d / eps^3, must not underflow).  At most
// 2^5 below max|x| all the same: the smallest pair terms, of the system's
// size, stay 2^32 above the grid (a VJP's or jerk's, which fall with its cube;
// kMaxBound), and an eps 2^47 below max|x|, where eps^-3 is infinite again, is
// at the 48 bits of the positions.
constexpr int kSmallEps = 36, kUnitBelow = 5;
__host__ __device__ constexpr int length_exponent(int ex, int ee) {
    int z = ex < ee + kSmallEps ? ex : ee + kSmallEps;
    z = z > ex - kUnitBelow ? z : ex - kUnitBelow;
    z = z > ee ? z : ee;
    return z < -60 ? -60 : (z > 60 ? 60 : z);
}
// Exponent of the scaled bounds at most: no finite FP32 partial is larger, and
// 2^19 of them fit the limbs.
constexpr int kMaxBound = 127;
// Where the packs put padding slots along x: their pairs must be finite (at the
// origin, zero mass times r^-3 at a particle on the same spot was a NaN), which
// they are between 2^-4 and 2^116 units of length.
constexpr float kPadX = 72057594037927936.f;  // 2^56
// Exponents of the maxima (v < 2^e; fx::kNoBound: not finite), for the bounds:
// integers, because a few dependent FP64 operations at the start of every
// kernel cost microseconds on this part.
struct Maxima {
    int m, v, c, p;
};
enum Factor { kFx = 0, kFm = 1, kFc = 2, kFp = 3, kFone = 4 };  // 2^-x 2^-m 2^-c 2^(x - c)

// e with v < 2^e for the float with these bits (0 for 0, inf and NaN), within
// +-60, so that every factor is a normal float.
__device__ __forceinline__ int exponent_of(unsigned bits) {
    const int f = (int)(bits >> 23);
    return f == 0 || f == 0xff ? 0 : min(max(f - 126, -60), 60);
}
__device__ __forceinline__ int exponent_or(unsigned bits, int other) {
    const int f = (int)(bits >> 23);
    return f == 0 || f == 0xff ? other : f - 126;
}
__device__ __forceinline__ int bound_exponent(unsigned bits) {
    const int f = (int)(bits >> 23);
    return f == 0xff ? fx::kNoBound : f == 0 ? -126 : f - 126;
}
__device__ __forceinline__ float pow2f(int e) { return __uint_as_float((unsigned)(127 + e) << 23); }

// Folds the warp's largest |v| into a max word (all 32 lanes call it).
__device__ __forceinline__ void warp_max(unsigned *word, float v) {
    const unsigned b = __reduce_max_sync(0xffffffffu, __float_as_uint(v));
    if ((threadIdx.x & 31) == 0 && b) atomicMax(word, b);
}

// Row I of the triangular item list starts at item row_start(I).
__host__ __device__ __forceinline__ int64_t row_start(int64_t I, int64_t nb) {
    return I * nb - I * (I - 1) / 2;
}

// Item t's blocks (I, J).  The discriminant is an exact integer; the float
// square root is off by at most a row, which the two loops repair.
__host__ __device__ __forceinline__ void item_of(int64_t t, int64_t nb, int &I, int &J) {
    const int64_t b = 2 * nb + 1;
    int64_t r = (int64_t)(((float)b - sqrtf((float)(b * b - 8 * t))) * 0.5f);
    r = r < 0 ? 0 : (r > nb - 1 ? nb - 1 : r);
    while (r > 0 && row_start(r, nb) > t) --r;
    while (r + 1 < nb && row_start(r + 1, nb) <= t) ++r;
    I = (int)r;
    J = (int)(r + (t - row_start(r, nb)));
}

__device__ __forceinline__ void poison(unsigned long long *top_limb) {
    atomicMax(reinterpret_cast<long long *>(top_limb), fx::kPoison);
}

// TwoSum (Knuth): a + b as a float and its exact rounding error.
__device__ __forceinline__ float2 two_sum(float a, float b) {
    const float s = __fadd_rn(a, b);
    const float z = __fsub_rn(s, a);
    return f2(s, __fadd_rn(__fsub_rn(a, __fsub_rn(s, z)), __fsub_rn(b, z)));
}
// t + x as an unevaluated pair; without `keep` (the FP32 policy's plain running
// sums) the rounding error of the add is dropped.
__device__ __forceinline__ float2 two_add(float2 t, float x, bool keep = true) {
    const float2 u = two_sum(t.x, x);
    return f2(u.x, keep ? __fadd_rn(t.y, u.y) : 0.f);
}

// A row's running total of a component over a warp's segment and the warps of
// a CTA.  KAHAN: a compensated float pair; FP32: a plain float (keep = false).
template <bool F64>
struct Total {
    float2 v;
    __device__ __forceinline__ void zero() { v = f2(0.f, 0.f); }
    __device__ __forceinline__ void add(float x, bool keep) { v = two_add(v, x, keep); }
    __device__ __forceinline__ void merge(const Total &o) { v = two_add(two_add(v, o.v.x), o.v.y); }
    // the floats to add up; the low ones are zero for the first flushes of a row
    template <class F>
    __device__ __forceinline__ void parts(const F &f) const {
        f(v.x);
        if (v.y != 0.f) f(v.y);
    }
};
// F64ACC and the VJP: three floats, s and c by TwoSum, so that only additions
// into d round, 2^-48 below the total: more than the 53 bits of the FP64 sums
// that they stand for, in 13 FP32 operations.  An FP64 add holds the pipe of
// this part for as long as 64 of them.  Against a float pair for F64ACC too:
// 433 us a step at 32768 with the pair, 444 in FP64, 434 so; acceleration +
// jerk 779 / 863 / 779 us; VJP of 16384 195.0 / 200.2 / 198.4 us.
template <>
struct Total<true> {
    float s, c, d;
    __device__ __forceinline__ void zero() { s = c = d = 0.f; }
    __device__ __forceinline__ void add(float x, bool = true) {
        const float2 t = two_sum(s, x), u = two_sum(c, t.y);
        s = t.x;
        c = u.x;
        d = __fadd_rn(d, u.y);
    }
    __device__ __forceinline__ void merge(const Total &o) {
        const float2 t = two_sum(s, o.s), u = two_sum(c, o.c), v = two_sum(u.x, t.y);
        s = t.x;
        c = v.x;
        d = __fadd_rn(d, __fadd_rn(o.d, __fadd_rn(u.y, v.y)));
    }
    template <class F>
    __device__ __forceinline__ void parts(const F &f) const {
        f(s);
        if (c != 0.f) f(c);
        if (d != 0.f) f(d);
    }
};

// Geometry of a physics: K register groups per lane.  With IPAIR a group's .x
// and .y are two i-slots and the lane has one j-particle, broadcast as (x, x);
// otherwise a group is one i-slot, broadcast, and .x and .y are two j.
template <class PH>
struct Geo {
    static constexpr int SL = PH::IPAIR ? 2 * PH::K : PH::K;  // i-slots per lane
    static constexpr int JL = PH::IPAIR ? 1 : 2;              // j-slots per lane
    static constexpr int BW = 32 * SL;                        // slots per block
    static constexpr int JSET = 32 * JL;                      // slots per j-set
    static constexpr int JPB = BW / JSET;                     // j-sets per block
    static constexpr int UPJ = 32 / GR, UPI = JPB * UPJ;      // scheduling units
    static constexpr int NV = SL * PH::NC, NTHR = 32 * PH::WARPS;
    static_assert(2048 % BW == 0 && BW >= kMinBlockSlots, "blocks tile the padded pack");
};

// Zeroes the halves of v that pair a particle with itself: rotation step 0 of
// the diagonal block's j-set h.  What is zeroed is r^-1, so that nothing
// infinite meets a zero.
template <bool IPAIR>
__device__ __forceinline__ float2 mask_self(float2 v, int k, int h) {
    v.x = (IPAIR ? h == 2 * k : k == 2 * h) ? 0.f : v.x;
    v.y = (IPAIR ? h == 2 * k + 1 : k == 2 * h + 1) ? 0.f : v.y;
    return v;
}

__device__ __forceinline__ float2 neg(float2 v) { return f2(-v.x, -v.y); }

// i-side values that few operations use: a scalar broadcast at the use, or
// with IPAIR the pair itself.
template <bool IPAIR>
using LoT = std::conditional_t<IPAIR, float2, float>;
template <bool IPAIR>
__device__ __forceinline__ LoT<IPAIR> lo_of(float2 v) {
    if constexpr (IPAIR)
        return v;
    else
        return v.x;
}
__device__ __forceinline__ float2 lo2(float v) { return f2(v, v); }
__device__ __forceinline__ float2 lo2(float2 v) { return v; }

// n rotation steps of one j-set; B: the j-particles' sums (IPAIR: in .x).
template <class PH, bool SYM>
__device__ __forceinline__ void rotate(typename PH::S &S, const float2 e2,
                                       const float (&j)[Geo<PH>::JL * PH::NJ],
                                       float2 (&B)[PH::NC], const int n, const int self_h) {
    constexpr bool IP = PH::IPAIR;
    const int src = (threadIdx.x + 1) & 31;
    float2 J[PH::NJ];
#pragma unroll
    for (int a = 0; a < PH::NJ; ++a) J[a] = f2(j[a], IP ? j[a] : j[(Geo<PH>::JL - 1) * PH::NJ + a]);
#pragma unroll
    for (int e = 0; e < PH::NC; ++e) B[e] = f2(0.f, 0.f);
    auto down = [&](float2 v) {
        const float x = __shfl_sync(0xffffffffu, v.x, src);
        return f2(x, IP ? x : __shfl_sync(0xffffffffu, v.y, src));
    };
    // the shuffles for the next step go out before this step's arithmetic,
    // which hides their latency; the sums therefore lag one lane behind
    auto one = [&](auto self) {
        float2 Jn[PH::NJ], T[PH::NC];
#pragma unroll
        for (int a = 0; a < PH::NJ; ++a) Jn[a] = down(J[a]);
        if (SYM) {
#pragma unroll
            for (int e = 0; e < PH::NC; ++e) B[e] = down(B[e]);
        }
        PH::template step<SYM, decltype(self)::value>(S, e2, J, T, self_h);
        if (SYM) {
#pragma unroll
            for (int e = 0; e < PH::NC; ++e)
                B[e] = IP ? f2(__fadd_rn(B[e].x, __fadd_rn(T[e].x, T[e].y)), 0.f)
                          : f2(__fadd_rn(B[e].x, T[e].x), __fadd_rn(B[e].y, T[e].y));
        }
#pragma unroll
        for (int a = 0; a < PH::NJ; ++a) J[a] = Jn[a];
    };
    int st = 0;
    if (!SYM && self_h >= 0) {
        one(std::true_type{});
        st = 1;
    }
#pragma unroll 2
    for (; st < n; ++st) one(std::false_type{});
}

template <class PH>
__device__ __forceinline__ void load_j(const Params &p, int slot,
                                       float (&j)[Geo<PH>::JL * PH::NJ]) {
#pragma unroll
    for (int a = 0; a < PH::NJ; ++a) {
        const float *q = PH::plane(p, a) + slot;
#pragma unroll
        for (int h = 0; h < Geo<PH>::JL; ++h) j[h * PH::NJ + a] = q[32 * h];
    }
}

template <class PH, bool F64>
__global__ void __launch_bounds__(Geo<PH>::NTHR, 1) wsym_kernel(const Params p) {
    using GE = Geo<PH>;
    constexpr int NWARP = PH::WARPS, NTHR = GE::NTHR, NC = PH::NC, NV = GE::NV;
    constexpr int BW = GE::BW, JSET = GE::JSET, UPJ = GE::UPJ, UPI = GE::UPI;
    extern __shared__ __align__(16) unsigned char wsym_smem[];
    using Tot = Total<F64>;
    Tot *tot = reinterpret_cast<Tot *>(wsym_smem);  // [NV][NTHR]
    __shared__ int sF[kMaxGroups];
    __shared__ int stag[NWARP];
    __shared__ float sFac[4];
    const int tid = threadIdx.x, w = tid >> 5, l = tid & 31;
    // the first `extra` warps take one unit more than the others
    const int64_t gw = (int64_t)blockIdx.x * NWARP + w;
    int64_t u = gw * p.per_warp + (gw < p.extra ? gw : p.extra);
    const int64_t u_end = u + p.per_warp + (gw < p.extra ? 1 : 0);
    const int nslots = (int)(p.nb * BW);
    uint32_t bad = 0;
    int I = 0, jb = 0, tag = -1;
    if (u < u_end) {
        int J;
        item_of(u / UPI, p.nb, I, J);
        jb = J * BW + (int)(u % UPI) / UPJ * JSET;
    }
    // no grid_trigger(): placing the fold's blocks while this kernel fills the
    // SMs cost 10 us a step (2047: 21.8 / 11.6 us, 16384: 128.6 / 117.6 us)
    dev::grid_wait();
    if (w == 0) {
        const unsigned bx = __ldcg(p.mx + kMaxX), bm = __ldcg(p.mx + kMaxM),
                       bv = __ldcg(p.mx + kMaxV), bc = __ldcg(p.mx + kMaxC),
                       bp = __ldcg(p.mx + kMaxP);
        Scales z;
        const int ee = exponent_or(__float_as_uint(p.eps), 60);
        z.x = length_exponent(exponent_or(bx, ee), ee);
        z.m = exponent_of(bm);
        z.c = min(max(exponent_of(bc), exponent_of(bp) + z.x), 60);
        const Maxima mm = {bound_exponent(bm), bound_exponent(bv), bound_exponent(bc),
                           bound_exponent(bp)};
        if (l < PH::GROUPS) {
            const int up = PH::shift(z, l);
            const int b = PH::bound(p, mm, l) - up;
            const int Fg = fx::limb_exponent(b >= fx::kNoBound / 2 ? b : min(b, kMaxBound));
            sF[l] = Fg;
            // value = 2^up (scaled value)
            if (blockIdx.x == 0) p.fxe[l] = Fg == fx::kNoGrid ? Fg : Fg - up;
        }
        if (l == 0) {
            sFac[kFx] = pow2f(-z.x);
            sFac[kFm] = pow2f(-z.m);
            sFac[kFc] = pow2f(-z.c);
            sFac[kFp] = pow2f(z.x - z.c);
        }
    }
    __syncthreads();
    // eps^2 in scaled lengths (at least the smallest normal float)
    const float eu = p.eps * sFac[kFx], es = fmaxf(eu * eu, 1.17549435e-38f);
    const float2 e2 = f2(es, es);
    int F[PH::GROUPS];
#pragma unroll
    for (int g = 0; g < PH::GROUPS; ++g) F[g] = sF[g];
    typename PH::S S;
    float jn[GE::JL * PH::NJ];
    bool open = false;
    int pend = 0;
    auto flush_regs = [&]() {
#pragma unroll
        for (int k = 0; k < PH::K; ++k)
#pragma unroll
            for (int e = 0; e < NC; ++e) {
                if constexpr (PH::IPAIR) {
                    Tot *t = tot + (2 * k * NC + e) * NTHR + tid;
                    t->add(S.a[k][e].x, p.keep);
                    t[NC * NTHR].add(S.a[k][e].y, p.keep);
                } else {
                    tot[(k * NC + e) * NTHR + tid].add(S.a[k][e].x + S.a[k][e].y, p.keep);
                }
                S.a[k][e] = f2(0.f, 0.f);
            }
        pend = 0;
    };
    auto add = [&](int e, int slot, float v, int Fe) {
        int q;
        long long lo, hi;
        const bool ok = fx::split_limbs(v, Fe, q, lo, hi);
        if (slot >= p.N) return;
        unsigned long long *wd = p.fx + (int64_t)(fx::kLimbs * e + q) * p.Np + slot;
        if (!ok) {
            bad = 1;
            poison(wd + (fx::kLimbs - 1) * p.Np);  // q is 0
        }
        if (lo) atomicAdd(wd, (unsigned long long)lo);
        if (hi) atomicAdd(wd + p.Np, (unsigned long long)hi);
    };
    auto add_row = [&](int e, int slot, const Tot &t) {
        t.parts([&](float v) { add(e, slot, v, sF[PH::group(e)]); });
    };
    while (u < u_end) {
        const int r0 = (int)u & (UPJ - 1), s0 = r0 * GR;
        const int un = u_end - u < UPJ - r0 ? (int)(u_end - u) : UPJ - r0;
        if (!open) {
#pragma unroll
            for (int k = 0; k < PH::K; ++k) {
                float2 v[PH::NJ];
#pragma unroll
                for (int a = 0; a < PH::NJ; ++a) {
                    const float *q = PH::plane(p, a) + I * BW + (PH::IPAIR ? 64 : 32) * k + l;
                    const float fa = PH::factor(a) == kFone ? 1.f : sFac[PH::factor(a)];
                    v[a].x = q[0] * fa;
                    v[a].y = PH::IPAIR ? q[32] * fa : v[a].x;
                }
                PH::set_i(S, k, v);
#pragma unroll
                for (int e = 0; e < NC; ++e) S.a[k][e] = f2(0.f, 0.f);
            }
#pragma unroll
            for (int v = 0; v < NV; ++v) tot[v * NTHR + tid].zero();
            load_j<PH>(p, jb + ((l + s0) & 31), jn);
            open = true;
        }
        float jc[GE::JL * PH::NJ];
#pragma unroll
        for (int a = 0; a < GE::JL * PH::NJ; ++a) {  // scaled here: the prefetch must not wait
            const int fa = PH::factor(a % PH::NJ);
            jc[a] = fa == kFone ? jn[a] : jn[a] * sFac[fa];
        }
        u += un;
        const int jnext = jb + JSET;
        const bool row_end = jnext >= nslots;
        if (u < u_end && !row_end) load_j<PH>(p, jnext + l, jn);
        float2 B[NC];
        const int n = un * GR;
        if (jb >= (I + 1) * BW) {
            rotate<PH, true>(S, e2, jc, B, n, -1);
            const int js = jb + ((l + s0 + n - 1) & 31);
#pragma unroll
            for (int e = 0; e < NC; ++e) {
#pragma unroll
                for (int h = 0; h < GE::JL; ++h) {
                    const float v = h ? B[e].y : B[e].x;
                    add(e, js + 32 * h, PH::jneg(e) ? -v : v, F[PH::group(e)]);
                }
            }
        } else {
            rotate<PH, false>(S, e2, jc, B, n, s0 == 0 ? (jb - I * BW) / JSET : -1);
        }
        const bool end = u >= u_end;
        if (++pend == FLUSH || row_end || end) flush_regs();
        if (end) {
            tag = I;
        } else if (row_end) {
#pragma unroll 1
            for (int v = 0; v < NV; ++v)
                add_row(v % NC, I * BW + 32 * (v / NC) + l, tot[v * NTHR + tid]);
            ++I;
            jb = I * BW;
            open = false;
        } else {
            jb = jnext;
        }
    }
    // the warps' last segments, row by row over the CTA
    if (l == 0) stag[w] = tag;
    __syncthreads();
#pragma unroll 1
    for (int v = tid; v < NV * 32; v += NTHR) {
        const int vk = v >> 5, lane = v & 31, e = vk % NC, k = vk / NC;
        Tot t;
        t.zero();
        int row = -1;
#pragma unroll 1
        for (int w2 = 0; w2 <= NWARP; ++w2) {
            const int r = w2 < NWARP ? stag[w2] : -1;
            if (r != row) {
                if (row >= 0) add_row(e, row * BW + 32 * k + lane, t);
                t.zero();
                row = r;
            }
            if (r >= 0) t.merge(tot[vk * NTHR + 32 * w2 + lane]);
        }
    }
    if (bad) dev::set_status(p.status, kStatusNonFinite);
}

// The fold leaves the totals that it reads at zero, but the workspace may have
// served another size or kernel since: the pack of every call makes sure, with
// blocks of 128 threads beyond the ones that pack the slots, a component of two
// slots per thread.  They read first: stores that have to be out before the
// pair kernel cost more than the loads, which the pack's own hide (acceleration
// + jerk of 1024 particles: 18.8 us with totals known to be zero and so, 20.4
// us when the packing threads stored the 24 words of a particle).
inline unsigned pack_blocks(int64_t slots, int64_t N, int nc) {
    return (unsigned)(cdiv(slots, 128) + nc * cdiv(N, 256));
}
// True for the clearing blocks, after their work.
__device__ __forceinline__ bool clear_totals(unsigned long long *fx, int64_t slots, int64_t N,
                                             int64_t Np, int nc) {
    const int b = (int)(blockIdx.x - (unsigned)((slots + 127) / 128));
    if (b < 0) return false;
    const int64_t s = 2 * ((int64_t)(b / nc) * 128 + threadIdx.x);  // Np is even
    if (s < N) {
        unsigned long long *q = fx + (int64_t)(b % nc) * fx::kLimbs * Np + s;
        ulonglong2 v[fx::kLimbs];
#pragma unroll
        for (int k = 0; k < fx::kLimbs; ++k) v[k] = *reinterpret_cast<const ulonglong2 *>(q + k * Np);
#pragma unroll
        for (int k = 0; k < fx::kLimbs; ++k)
            if (v[k].x | v[k].y)
                *reinterpret_cast<ulonglong2 *>(q + k * Np) = make_ulonglong2(0ull, 0ull);
    }
    return true;
}

// Reads and zeroes component e of slot s; its value.
__device__ __forceinline__ double take_fixed(const Params &p, int e, int64_t s, int F) {
    unsigned long long *wd = p.fx + (int64_t)(fx::kLimbs * e) * p.Np + s;
    long long w[fx::kLimbs];
#pragma unroll
    for (int q = 0; q < fx::kLimbs; ++q) w[q] = (long long)__ldcs(wd + q * p.Np);
#pragma unroll
    for (int q = 0; q < fx::kLimbs; ++q)
        if (w[q]) wd[q * p.Np] = 0ull;
    return fx::limb_value(w, F);
}

// One CTA per SM, every warp the same number of steps.
template <class PH, bool F64>
int launch_pairs(Params &p, cudaStream_t st) {
    auto kern = wsym_kernel<PH, F64>;
    using GE = Geo<PH>;
    constexpr size_t smem = (size_t)GE::NV * GE::NTHR * sizeof(Total<F64>);
    const int rc = smem_optin(reinterpret_cast<const void *>(kern), smem);
    if (rc != NB_OK) return rc;
    p.nb = cdiv(p.N, GE::BW);
    const int64_t units = p.nb * (p.nb + 1) / 2 * GE::UPI;
    const int64_t ctas = std::min<int64_t>(device_sm_count(), cdiv(units, PH::WARPS));
    p.per_warp = units / (ctas * PH::WARPS);
    p.extra = units % (ctas * PH::WARPS);
    return launch_pdl(kern, (unsigned)ctas, GE::NTHR, smem, st, p);
}

}  // namespace wsym
}  // namespace nb
