// Symmetric-pair force evaluation (Eq. 1 with Newton's third law).
//
// The pair term of Eq. 1 is antisymmetric up to the masses: with
// d = x_j - x_i and r^-3 = (|d|^2 + eps^2)^-3/2,
//     a_i += m_j r^-3 d,   a_j -= m_i r^-3 d,
//     phi_i += m_j r^-1,   phi_j += m_i r^-1,
// so one evaluation of d, r^2, r^-1 and r^-3 serves both particles.  Per
// unordered pair that is 18 FP32 operations (single-float displacement) in
// place of 2 x 13, about 9 per directed interaction.
//
// Decomposition.  The (padded) slots are cut into row blocks of 2048; the
// work items are the block pairs (I, J) with J >= I, in row-major order,
// cut into units of 2 j-sets and split over one persistent CTA per SM into
// contiguous ranges of equal estimated cost (stream-K: a range may start or
// end inside an item).  The estimate counts FP32 operations per (warp,
// j-set) from the same near/far box tests the pair kernel makes; three small
// kernels compute it, scan it and cut the ranges.
// A CTA of 8 warps keeps block I in registers: warp w holds the 256 slots
// I*2048 + w*256 + [0, 256), lane l the eight slots  + 32k + l  (k = 0..7),
// each pre-broadcast as an (x, x) pair.  A j-set is 64 slots of block J;
// lane l loads two of them, j-slots l and 32 + l, into the .x / .y halves
// of packed f32x2 registers, so every FP32 operation of the pair term is a
// packed one (one rotation step: 8 i-slots x 2 j = 16 pairs, 148 packed
// FP32 instructions, 16 MUFU rsqrt, 16 shuffles).  The set rotates through
// the lanes with shuffles: at step s lane l holds j-slots (l + s) mod 32 and
// 32 + (l + s) mod 32, so in 32 steps every lane meets every j once, and the
// j-particles' own sums (a_j, phi_j) travel with them and come home to lane
// l.  Each step's eight j-side terms go into fresh registers and then into
// the travelling sums with one add, so a strong close pair's term meets
// ~47 later FP32 roundings within an item, not ~260.
//
//   * Off-diagonal items (I < J): both halves of every pair.  The 8 warps'
//     j-side sums of 2 j-sets are added in warp order in shared memory (one
//     barrier per 2 j-sets), giving the FP32 partial of the J-block
//     particles from block I.
//   * Diagonal items (I = J): the i-side only, over all ordered pairs of
//     the block; the self pairs (j-set 4w + h at rotation step 0: i-slot 2h
//     against the .x j, 2h + 1 against the .y j) get a zero mass, so Eq. 1's
//     j != i holds exactly.
//
// The i-side FP32 register sums, kept per j-stream (.x, .y), are folded into
// the accumulation policy (FP32, Kahan or FP64; totals kept in shared
// memory) every 4 j-sets (128 terms per stream and particle; for F64ACC
// through an FP32 middle sum in shared memory that goes into FP64 every 8
// j-sets, FP64 adds being slow on this part) over the CTA's segment of a
// row.  In Hilbert order a particle's strongest, mutually cancelling terms
// (its spatial neighbours) arrive together; with 512-term FP32 chains the
// running sums of central particles of a log-normal Plummer sphere
// (N = 300001, eps = 1e-3) lost up to 1e-5 of |a|, with 128-term chains they
// stay at the 2e-6 of the unsorted order.  (Flushing every 2 j-sets was
// measured 0.8 % slower at 2^20 for 2.08e-6 -> 1.94e-6 worst error.)
//
// Combining across CTAs.  Every particle's sum collects one j-side FP32
// partial per block above it and one i-side total per CTA that worked on its
// row.  Both go, as they are produced, into two-word fixed-point
// accumulators (nb_fixed.cuh) with integer atomic adds: exact and
// independent of arrival order, so results are bitwise reproducible, and the
// scratch is O(N) (64 B per particle) -- not a partial per block pair.  A
// one-block kernel picks the fixed-point exponent from the a-priori bound
// N max|m| max(0.385 / eps^2, 1 / eps) on every partial and total (the
// largest value of |d| (|d|^2 + eps^2)^-3/2 is 0.385 / eps^2 at
// |d| = eps / sqrt 2).  The fold kernel reads each particle's accumulators
// once (and zeroes them for a loop's next evaluation), applies G, scatters through the
// Hilbert permutation and optionally kicks the velocity.
//
// Displacements are adaptive: per (warp i-set, j-set) the hi/lo form
// (x_j.hi - x_i.hi) + (x_j.lo - x_i.lo) only when the bounding boxes are
// closer than gamma * max|x| (a 32-bit mask per warp and item, from the
// Hilbert-sorted pack's boxes of 256 i- and 64 j-slots), single floats
// elsewhere.  Systems with one form for every pair (single floats: MODE 0,
// hi/lo: MODE 1) are not sorted; below kSymPlainMinN they go to nb_wsym.cu,
// whose j-side sums are added to the totals per block of 128 or 256 slots
// instead of 2048 -- finer ranges, but 8 to 16 times the atomics, which no
// longer fit beside the arithmetic once the totals outgrow the L2 (MODE 0
// here / there: 1288 / 1346 us a step at 65536, 5.21 / 5.74 ms at 131072,
// 328 / 365 ms at 2^20).
#include <cuda_runtime.h>

#include <stdlib.h>

#include <algorithm>
#include <cmath>

#include "nb_device.cuh"
#include "nb_fixed.cuh"
#include "nb_internal.h"
#include "nb_sym_core.cuh"
#include "nb_symj.cuh"

namespace nb {

using dev::Acc;
using dev::add2;
using dev::f2;
using dev::fma2;
using dev::mul2;
using dev::rsqrt_approx;

namespace {

using namespace symcore;
using namespace symj;

#define NB_TRY_SYM(...)                \
    do {                               \
        const int rc_ = (__VA_ARGS__); \
        if (rc_ != NB_OK) return rc_;  \
    } while (0)

constexpr int BI = 2048;            // slots per row block
static_assert(BI == kSymBlock, "row block size");
constexpr int CPS = 1;              // resident CTAs per SM
constexpr int US = 16;              // stream-K units per item
constexpr int NW = 8;               // warps per CTA
constexpr int NT = NW * 32;         // threads per CTA
constexpr int IRP = 8;              // i-slots per lane
constexpr int WS = 32 * IRP;        // i-slots per warp
constexpr int JSP = 64;             // slots per j-set (two per lane)
constexpr int NJSP = BI / JSP;      // j-sets per block: one 32-bit near mask
constexpr int KBP = 2;              // j-sets per cross-warp reduction (128 slots)
constexpr int FLP = 4;              // j-sets per i-side flush (128 terms per j-stream)
constexpr int FL2P = 16;            // F64ACC: j-sets per FP64 add of the FP32 middle sums
                                    // (1024 pair terms; 8 j-sets: 341.4 ms at 2^20, 16: 334.5)
static_assert(NW * WS == BI && NJSP == 32 && NJSP / KBP == US, "FP32 kernel shape");
constexpr size_t kRedBytes = 2 * KBP * 2 * NW * 32 * sizeof(float4);
struct SymParams {
    const float *soa;   // packed SoA [7][Np]
    int64_t Np;
    int64_t nb;         // row blocks
    int64_t T;          // items nb (nb + 1) / 2
    int64_t U;          // stream-K units T * US (KBP j-sets of one item each)
    int64_t ctas;       // grid size of the pair kernel
    float eps2;
    int mode;           // displacement: 0 single floats, 1 hi/lo, 2 adaptive
    float gamma;        // adaptive threshold
    const float *jbox;  // per 64 slots: lo[3], hi[3], max|x|, pad
    const float *wbox;  // per 256 slots
    unsigned long long *acc_fx;  // [4 components][2 words][Np] fixed-point totals
    const int *fx_exp;           // the call's fixed-point exponent F
    const int64_t *lo;  // [ctas + 1]: CTA c owns units [lo[c], lo[c + 1])
    uint32_t *status;
};

__host__ __device__ inline int64_t row_start(int64_t I, int64_t nb) {
    return I * nb - I * (I - 1) / 2;
}

// Adds v to component e of slot s's fixed-point total.
__device__ __forceinline__ void add_fixed(const SymParams &p, int e, int64_t s, double v, int F) {
    unsigned long long *w = p.acc_fx + (int64_t)(2 * e) * p.Np + s;
    if (!fx::add(w, w + p.Np, v, F)) dev::set_status(p.status, kStatusNonFinite);
}
__device__ __forceinline__ void add_fixed(const SymParams &p, int e, int64_t s, float v, int F) {
    unsigned long long *w = p.acc_fx + (int64_t)(2 * e) * p.Np + s;
    if (!fx::add_f32(w, w + p.Np, v, F)) dev::set_status(p.status, kStatusNonFinite);
}

// ------------------------------------------------------------- FP32 pairs
__device__ __forceinline__ void load_jp(const SymParams &p, int64_t s, float (&j)[14]) {
    symj::load_pair(p.soa, p.Np, s, j);
}

// POT: the potential sums too (the caller wants phi).  The i-slots' lo parts
// stay in registers for MODE 1 (every j-set is near) and come from shared
// memory for MODE 2 (only near j-sets use them, and 245 of 255 registers are
// taken).
template <int POL, int MODE, bool POT>
__global__ void __launch_bounds__(NT, CPS) force_sym_kernel(const SymParams p) {
    constexpr int NWJ = NW, IRJ = IRP, SNTJ = NT;
    constexpr bool LOSM = MODE == 2;
    constexpr int HW = IRJ / 2;  // j-sets per warp i-set
    constexpr size_t kRedBytesJ = kRedBytes;
    extern __shared__ __align__(16) unsigned char smemj[];
    float4 *red = reinterpret_cast<float4 *>(smemj);  // [2][KBP][2 halves][NWJ][32]
    Acc<POL> *tot = reinterpret_cast<Acc<POL> *>(smemj + kRedBytesJ);  // [IRJ * 4][SNTJ]
    constexpr bool MID = POL == NB_PREC_F64ACC;
    float *mid = reinterpret_cast<float *>(smemj + kRedBytesJ + 4 * IRJ * SNTJ * sizeof(Acc<POL>));
    // LOSM: (-x.lo, -x.lo) pairs [3][IRJ][SNTJ] after the F64ACC middle sums
    float2 *lo2 = reinterpret_cast<float2 *>(smemj + kRedBytesJ +
                                             4 * IRJ * SNTJ * sizeof(Acc<POL>) +
                                             (MID ? 4 * IRJ * SNTJ * sizeof(float) : 0)) +
                  threadIdx.x;
    const int tid = threadIdx.x, w = tid >> 5, l = tid & 31;
    const int64_t c = blockIdx.x;
    int64_t u = __ldg(p.lo + c);
    const int64_t u_end = __ldg(p.lo + c + 1);
    if (u >= u_end) return;
    const int F = __ldg(p.fx_exp);
    const int64_t t0 = u / US;
    int64_t I = 0;
    while (row_start(I + 1, p.nb) <= t0) ++I;
    int64_t J = I + (t0 - row_start(I, p.nb));
    const float2 e2 = f2(p.eps2, p.eps2);
    ISetJ<IRJ> S;
    int half = 0;
    bool row_open = false;
    while (u < u_end) {
        const int qa = (int)(u % US) * KBP;
        const int64_t item_end = (u / US + 1) * US;
        const int64_t seg_end = item_end < u_end ? item_end : u_end;
        const int qb = qa + (int)(seg_end - u) * KBP;
        const int64_t ib = I * BI + w * (32 * IRJ);  // this warp's i-set
        if (!row_open) {
#pragma unroll
            for (int k = 0; k < IRJ; ++k) {
                const int64_t sl = ib + 32 * k + l;
                const float x = __ldg(p.soa + sl), y = __ldg(p.soa + p.Np + sl),
                            z = __ldg(p.soa + 2 * p.Np + sl), m = __ldg(p.soa + 3 * p.Np + sl);
                S.nx[k] = f2(-x, -x);
                S.ny[k] = f2(-y, -y);
                S.nz[k] = f2(-z, -z);
                S.m[k] = f2(m, m);
                const float xl = __ldg(p.soa + 4 * p.Np + sl), yl = __ldg(p.soa + 5 * p.Np + sl),
                            zl = __ldg(p.soa + 6 * p.Np + sl);
                if (LOSM) {
                    lo2[(0 * IRJ + k) * SNTJ] = f2(-xl, -xl);
                    lo2[(1 * IRJ + k) * SNTJ] = f2(-yl, -yl);
                    lo2[(2 * IRJ + k) * SNTJ] = f2(-zl, -zl);
                } else {
                    S.nxl[k] = -xl;
                    S.nyl[k] = -yl;
                    S.nzl[k] = -zl;
                }
                S.ax[k] = S.ay[k] = S.az[k] = S.ph[k] = f2(0.f, 0.f);
            }
#pragma unroll
            for (int v = 0; v < 4 * IRJ; ++v) {
                tot[v * SNTJ + tid].zero();
                if (MID) mid[v * SNTJ + tid] = 0.f;
            }
            row_open = true;
        }
        const bool sym = J != I;
        const int64_t jb = J * BI;
        unsigned near = 0u;
        if (MODE == 2) {
            float wb[7], tb[7];
#pragma unroll
            for (int a = 0; a < 7; ++a) {
                wb[a] = __ldg(p.wbox + (ib / (32 * IRJ)) * 8 + a);
                tb[a] = __ldg(p.jbox + (jb / JSP + l) * 8 + a);
            }
            near = __ballot_sync(0xffffffffu, boxes_near(wb, tb, p.gamma));
        }
        float jn[14];
        load_jp(p, jb + qa * JSP + l, jn);
        for (int q = qa; q < qb; ++q) {
            float jc[14];
#pragma unroll
            for (int a = 0; a < 14; ++a) jc[a] = jn[a];
            if (q + 1 < qb) load_jp(p, jb + (q + 1) * JSP + l, jn);
            const bool nq = (near >> q) & 1u;
            float4 b0, b1;
            if (sym) {
                run_setj<IRJ, MODE, true, POT, LOSM>(S, e2, jc, nq, b0, b1, -1, lo2, SNTJ);
                float4 *r = red + (((half * KBP + (q % KBP)) * 2) * NWJ + w) * 32 + l;
                r[0] = b0;
                r[NWJ * 32] = b1;
            } else {
                // the warp's own slots are j-sets HW w .. HW w + HW - 1 of the block
                run_setj<IRJ, MODE, false, POT, LOSM>(S, e2, jc, nq, b0, b1,
                                          q / HW == w ? q % HW : -1, lo2, SNTJ);
            }
            if ((q + 1) % FLP == 0 || q + 1 == qb) {
#pragma unroll
                for (int k = 0; k < IRJ; ++k) {
                    const float2 v4[4] = {S.ax[k], S.ay[k], S.az[k], S.ph[k]};
#pragma unroll
                    for (int e = 0; e < 4; ++e) {
                        const int v = (k * 4 + e) * SNTJ + tid;
                        const float val = v4[e].x + v4[e].y;
                        if (MID)
                            mid[v] += val;
                        else
                            tot[v].add(val);
                    }
                    S.ax[k] = S.ay[k] = S.az[k] = S.ph[k] = f2(0.f, 0.f);
                }
                if (MID && ((q + 1) % FL2P == 0 || q + 1 == qb)) {
#pragma unroll
                    for (int v = 0; v < 4 * IRJ; ++v) {
                        tot[v * SNTJ + tid].add(mid[v * SNTJ + tid]);
                        mid[v * SNTJ + tid] = 0.f;
                    }
                }
            }
            if (sym && (q + 1) % KBP == 0) {
                __syncthreads();
                for (int v = tid; v < KBP * JSP * 4; v += SNTJ) {
                    const int e = v & 3, js = (v >> 2) & (JSP - 1), qq = v >> 8;
                    const float *r = reinterpret_cast<const float *>(
                                         red + (((half * KBP + qq) * 2 + (js >> 5)) * NWJ) * 32 +
                                         (js & 31)) + e;
                    float sum = 0.f;
#pragma unroll
                    for (int w2 = 0; w2 < NWJ; ++w2) sum += r[w2 * 32 * 4];
                    if (POT || e < 3)
                        add_fixed(p, e, jb + (q + 1 - KBP + qq) * JSP + js, e < 3 ? -sum : sum, F);
                }
                half ^= 1;
            }
        }
        u = seg_end;
        if ((J == p.nb - 1 && qb == NJSP) || u == u_end) {
#pragma unroll
            for (int k = 0; k < IRJ; ++k) {
                const int64_t slot = ib + 32 * k + l;
#pragma unroll
                for (int e = 0; e < 4; ++e)
                    if (POT || e < 3) add_fixed(p, e, slot, tot[(k * 4 + e) * SNTJ + tid].value(), F);
            }
            row_open = false;
        }
        if (qb == NJSP && ++J == p.nb) {
            ++I;
            J = I;
        }
    }
}

// Reads and zeroes every slot's fixed-point totals (padding slots too: they
// collect j-side sums as zero-mass test particles); for real particles,
// applies G, writes acc / pot through the permutation (NULL = identity) and
// optionally kicks the velocity.
__global__ void __launch_bounds__(256) sym_fold_kernel(const SymParams p, int64_t N,
                                                       const int *__restrict__ perm, double G,
                                                       double *__restrict__ acc,
                                                       double *__restrict__ pot,
                                                       double *__restrict__ vel, double kick) {
    const int F = __ldg(p.fx_exp);
    uint32_t bad = 0;
    for (int64_t s = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; s < p.Np;
         s += (int64_t)gridDim.x * blockDim.x) {
        double a[4];
#pragma unroll
        for (int e = 0; e < 4; ++e) {
            unsigned long long *wd = p.acc_fx + (int64_t)(2 * e) * p.Np + s;
            const unsigned long long hi = __ldcs(wd), lo = __ldcs(wd + p.Np);
            if (hi) wd[0] = 0ull;
            if (lo) wd[p.Np] = 0ull;
            a[e] = fx::value(hi, lo, F);
        }
        if (s >= N) continue;
        const double ax = G * a[0], ay = G * a[1], az = G * a[2];
        const double gp = -G * a[3];
        const int64_t i = perm ? (int64_t)perm[s] : s;
        acc[3 * i] = ax;
        acc[3 * i + 1] = ay;
        acc[3 * i + 2] = az;
        if (vel) {
            vel[3 * i] += kick * ax;
            vel[3 * i + 1] += kick * ay;
            vel[3 * i + 2] += kick * az;
        }
        if (pot) pot[i] = gp;
        if (!(isfinite(ax) && isfinite(ay) && isfinite(az) && isfinite(gp))) bad = 1;
    }
    if (bad) dev::set_status(p.status, kStatusNonFinite);
}

// Order-preserving image of a float as a signed integer, and back.
__device__ __forceinline__ int ordered_f(float x) {
    const int b = __float_as_int(x);
    return b >= 0 ? b : b ^ 0x7fffffff;
}
__device__ __forceinline__ float from_ordered_f(int b) {
    return __int_as_float(b >= 0 ? b : b ^ 0x7fffffff);
}

__device__ __forceinline__ void store_box(float *out, const float (&lo)[3], const float (&hi)[3]) {
    float amax = 0.f;
#pragma unroll
    for (int c = 0; c < 3; ++c) {
        out[c] = lo[c];
        out[3 + c] = hi[c];
        amax = fmaxf(amax, fmaxf(fabsf(lo[c]), fabsf(hi[c])));
    }
    out[6] = hi[0] < lo[0] ? 0.f : amax;  // no real slot: never near
    out[7] = 0.f;
}

// The fold of one step fused with the next one's opening where the Hilbert
// order is kept: the totals (read and zeroed) x G, this step's closing kick,
// the next one's opening kick and drift, the hi/lo pack of the new positions
// in place and the boxes of 64 and 256 slots (a block is 256 slots), as
// sym_fold_kernel, kick_drift_pack_kernel, pack_sorted_kernel and two
// slot_boxes_kernel launches do one after the other.  The acceleration is not
// stored: the next fold replaces it before anything reads it.  Not SORTED
// (MODE 0 and 1): particle order, no boxes.  At 65536
// particles the ten launches of a step besides the pair kernel took 76 us
// (ncu); now they are four, 28 us.
template <bool SORTED>
__global__ void __launch_bounds__(256) sym_fold_next_kernel(
    const SymParams p, int64_t N, const int *perm, double G, double *pos, double *vel, double kick,
    double next_kick, double drift, float *soa, float *jbox, float *wbox) {
    __shared__ int red[6][8];
    const int64_t s = blockIdx.x * (int64_t)256 + threadIdx.x;
    const int w = threadIdx.x >> 5, l = threadIdx.x & 31;
    dev::grid_trigger();
    dev::grid_wait();
    const int F = *p.fx_exp;
    unsigned long long wd[6];
#pragma unroll
    for (int k = 0; k < 6; ++k) wd[k] = p.acc_fx[(int64_t)k * p.Np + s];
#pragma unroll
    for (int k = 0; k < 6; ++k)
        if (wd[k]) p.acc_fx[(int64_t)k * p.Np + s] = 0ull;
    int lo[3] = {ordered_f(3e38f), ordered_f(3e38f), ordered_f(3e38f)};
    int hi[3] = {ordered_f(-3e38f), ordered_f(-3e38f), ordered_f(-3e38f)};
    if (s < N) {
        const int64_t i = SORTED ? (int64_t)perm[s] : s;
        bool ok = true;
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            const double a = G * fx::value(wd[2 * c], wd[2 * c + 1], F);
            ok = ok && isfinite(a);
            double v = vel[3 * i + c] + kick * a;
            v = v + next_kick * a;
            const double x = pos[3 * i + c] + drift * v;
            vel[3 * i + c] = v;
            pos[3 * i + c] = x;
            const float h = __double2float_rn(x);
            soa[c * p.Np + s] = h;
            soa[(4 + c) * p.Np + s] = __double2float_rn(x - (double)h);
            lo[c] = hi[c] = ordered_f(h);
        }
        if (!ok) dev::set_status(p.status, kStatusNonFinite);
    }
    if (!SORTED) return;
#pragma unroll
    for (int c = 0; c < 3; ++c) {
        lo[c] = __reduce_min_sync(0xffffffffu, lo[c]);
        hi[c] = __reduce_max_sync(0xffffffffu, hi[c]);
        if (l == 0) {
            red[c][w] = lo[c];
            red[3 + c][w] = hi[c];
        }
    }
    __syncthreads();
    if (threadIdx.x < 5) {  // four 64-slot boxes, then the block's
        const int w0 = threadIdx.x < 4 ? 2 * threadIdx.x : 0, nw = threadIdx.x < 4 ? 2 : 8;
        float bl[3], bh[3];
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            int a = red[c][w0], b = red[3 + c][w0];
            for (int k = 1; k < nw; ++k) {
                a = min(a, red[c][w0 + k]);
                b = max(b, red[3 + c][w0 + k]);
            }
            bl[c] = from_ordered_f(a);
            bh[c] = from_ordered_f(b);
        }
        store_box(threadIdx.x < 4 ? jbox + (4 * (int64_t)blockIdx.x + threadIdx.x) * 8
                                  : wbox + (int64_t)blockIdx.x * 8,
                  bl, bh);
    }
}

// The call's fixed-point exponent from the bound N max|m| max(0.385 / eps^2,
// 1 / eps) (x 1.02 for the rounding of FP32 partial sums) on every partial
// and total.  Every block takes the maximum of its share of the masses
// (independent loads, four per thread in flight) and folds it into one word
// with an integer atomicMax on the bits (non-negative doubles order like
// their bit patterns, so the maximum is exact and F reproducible); the last
// block to finish (arrival counter) computes F and resets both words.  The
// totals are cleared here too: the workspace may have served another size.
__global__ void __launch_bounds__(256) sym_exponent_kernel(const double *__restrict__ mass,
                                                           int64_t N, double eps,
                                                           int *__restrict__ F,
                                                           unsigned long long *mmax_bits,
                                                           unsigned *arrivals, ulonglong2 *totals,
                                                           int64_t ntotals) {
    __shared__ double part[8];
    __shared__ bool last;
    double m = 0.0;
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < ntotals; i += stride)
        totals[i] = make_ulonglong2(0ull, 0ull);
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < N; i += 4 * stride) {
        double v[4];
#pragma unroll
        for (int k = 0; k < 4; ++k) v[k] = i + k * stride < N ? fabs(__ldg(mass + i + k * stride)) : 0.0;
#pragma unroll
        for (int k = 0; k < 4; ++k) m = fmax(m, v[k]);
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) m = fmax(m, __shfl_xor_sync(0xffffffffu, m, o));
    if ((threadIdx.x & 31) == 0) part[threadIdx.x >> 5] = m;
    __syncthreads();
    if (threadIdx.x == 0) {
        for (int k = 1; k < 8; ++k) m = fmax(m, part[k]);
        atomicMax(mmax_bits, (unsigned long long)__double_as_longlong(m));
        __threadfence();
        last = atomicAdd(arrivals, 1u) == gridDim.x - 1;
    }
    __syncthreads();
    if (last && threadIdx.x == 0) {
        __threadfence();
        const double mm = __longlong_as_double((long long)atomicAdd(mmax_bits, 0ull));
        const double per = fmax(0.3849002 / (eps * eps), 1.0 / eps);
        *F = fx::exponent_for(1.02 * (double)N * mm * per);
        *mmax_bits = 0ull;
        *arrivals = 0u;
    }
}

// ------------------------------------------------ cost-weighted stream-K
// Relative cost of a stream-K unit (KBP j-sets of an item, at whose end
// the CTA's warps meet at a barrier): the slowest warp's FP32-pipe cycles
// per lane and step over the unit's j-sets -- far pairs 18 off the diagonal
// (13 on it: i-side only), near pairs 24 (19) -- plus 28 that every unit
// costs alike.  That constant was fitted to per-CTA timers: with 1 the CTAs'
// times grew with their number of units (regression slope ~40 % of a
// unit's mean time); with 28 the last CTA of a 2^20 Plummer evaluation ends
// 0.2 % after the mean (0.9 % with the earlier per-item sum of all warps'
// j-sets), of a 2^18 one 1.1 %.
constexpr uint32_t kCostSymFar = 18, kCostSymNear = 24, kCostDiagFar = 13, kCostDiagNear = 19;
constexpr uint32_t kCostSymUnit = 28;

__device__ __forceinline__ void item_of(int64_t t, int64_t nb, int64_t &I, int64_t &J) {
    const double b = 2.0 * (double)nb + 1.0;
    int64_t r = (int64_t)floor((b - sqrt(b * b - 8.0 * (double)t)) * 0.5);
    if (r < 0) r = 0;
    if (r > nb - 1) r = nb - 1;
    while (r > 0 && row_start(r, nb) > t) --r;
    while (r + 1 < nb && row_start(r + 1, nb) <= t) ++r;
    I = r;
    J = r + (t - row_start(r, nb));
}

// The near/far decisions the pair kernel will take on item t, by a warp: lane l
// takes j-set l (unit l / 2); a unit's cost, on its even lane, is the maximum
// over the warps of its two j-sets' sum (every one near or far unless the
// mode is adaptive).
__device__ __forceinline__ uint32_t unit_cost(const SymParams &p, int64_t t) {
    static_assert(NJSP == 32 && KBP == 2, "lane l: j-set l, unit l / 2");
    const int l = threadIdx.x & 31;
    int64_t I, J;
    item_of(t, p.nb, I, J);
    const bool sym = I != J;
    const uint32_t cn = sym ? kCostSymNear : kCostDiagNear;
    const uint32_t cf = sym ? kCostSymFar : kCostDiagFar;
    if (p.mode != 2) return (l & 1) ? 0u : 2 * (p.mode ? cn : cf) + kCostSymUnit;
    float tb[7];
#pragma unroll
    for (int a = 0; a < 7; ++a) tb[a] = p.jbox[(J * NJSP + l) * 8 + a];
    uint32_t m = 0;
    for (int w = 0; w < NW; ++w) {
        float wb[7];
#pragma unroll
        for (int a = 0; a < 7; ++a) wb[a] = p.wbox[(I * NW + w) * 8 + a];
        const uint32_t v = boxes_near(wb, tb, p.gamma) ? cn : cf;
        const uint32_t pair = v + __shfl_xor_sync(0xffffffffu, v, 1);
        m = pair > m ? pair : m;
    }
    return (l & 1) ? 0u : m + kCostSymUnit;
}

// One warp per item: the sum of its unit costs.
__global__ void __launch_bounds__(256) sym_cost_kernel(const SymParams p, uint32_t *cost) {
    const int64_t t = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5;
    dev::grid_trigger();
    dev::grid_wait();
    if (t >= p.T) return;  // whole warps
    uint32_t c = unit_cost(p, t);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) c += __shfl_xor_sync(0xffffffffu, c, o);
    if ((threadIdx.x & 31) == 0) cost[t] = c;
}

// One block: prefix[t] = sum of cost[0, t), prefix[T] = the total.
__global__ void __launch_bounds__(1024) sym_scan_kernel(const SymParams p, const uint32_t *cost,
                                                        unsigned long long *prefix) {
    __shared__ unsigned long long part[32];
    const int tid = threadIdx.x, w = tid >> 5, l = tid & 31;
    const int64_t per = (p.T + 1023) / 1024;
    const int64_t i0 = tid * per < p.T ? tid * per : p.T;
    const int64_t i1 = i0 + per < p.T ? i0 + per : p.T;
    dev::grid_trigger();
    dev::grid_wait();
    unsigned long long sum = 0;
    for (int64_t t = i0; t < i1; ++t) sum += cost[t];
    unsigned long long run = sum;  // inclusive scan over the warp, then the warps
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const unsigned long long v = __shfl_up_sync(0xffffffffu, run, o);
        if (l >= o) run += v;
    }
    if (l == 31) part[w] = run;
    __syncthreads();
    if (w == 0) {
        unsigned long long v = part[l];
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const unsigned long long x = __shfl_up_sync(0xffffffffu, v, o);
            if (l >= o) v += x;
        }
        part[l] = v;
    }
    __syncthreads();
    run += (w ? part[w - 1] : 0ull) - sum;
    for (int64_t t = i0; t < i1; ++t) {
        prefix[t] = run;
        run += cost[t];
    }
    if (tid == 0) prefix[p.T] = part[31];
}

// A warp per range start: lo[c] = the unit where the cumulative cost reaches c / ctas of the total
// (the nearest unit boundary, from the item's unit costs); lo[0] = 0,
// lo[ctas] = U, non-decreasing; the item by a search that probes 32 places at a
// time.  (A one-thread scan of the partial sums and one thread per range
// start, its search and its 256 box tests, took 31 us of a 65536-particle
// step.)
__global__ void __launch_bounds__(128) sym_ranges_kernel(const SymParams p,
                                                         const unsigned long long *prefix,
                                                         int64_t *lo) {
    const int l = threadIdx.x & 31;
    const int64_t c = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5;
    dev::grid_wait();
    if (c > p.ctas) return;  // whole warps
    if (c == 0 || c == p.ctas) {
        if (l == 0) lo[c] = c == 0 ? 0 : p.T * US;
        return;
    }
    const unsigned long long target = prefix[p.T] * (unsigned long long)c / (unsigned long long)p.ctas;
    int64_t a = 0, n = p.T;  // prefix[a] <= target; the item is one of n from a
    while (n > 1) {
        const int64_t st = (n + 31) / 32, t = a + l * st;
        const unsigned le =
            __ballot_sync(0xffffffffu, l * st < n && prefix[t < p.T ? t : p.T] <= target);
        const int h = 31 - __clz((int)le);  // lane 0 always holds
        n = n - h * st < st ? n - h * st : st;
        a += h * st;
    }
    const unsigned long long r = target - prefix[a];
    const uint32_t uc = unit_cost(p, a);
    unsigned long long acc = 0;
    int off = 0;
    for (int u = 0; u < US; ++u) {
        const uint32_t v = __shfl_sync(0xffffffffu, uc, 2 * u);
        if (off == u) {
            if (acc + v <= r) {
                acc += v;
                ++off;
            } else if (2 * (r - acc) > v) {
                off = u + 1;  // the nearer boundary
                break;
            } else {
                break;
            }
        }
    }
    if (l == 0) lo[c] = a * US + off;
}

template <int POL, int MODE, bool POT>
int launch_pair(const SymParams &p, cudaStream_t st) {
    auto kern = force_sym_kernel<POL, MODE, POT>;
    const size_t smem = kRedBytes + 4 * BI * sizeof(Acc<POL>) +
                        (POL == NB_PREC_F64ACC ? 4 * BI * sizeof(float) : 0) +
                        (MODE == 2 ? 3 * BI * sizeof(float2) : 0);
    const int rc = smem_optin(reinterpret_cast<const void *>(kern), smem);
    if (rc != NB_OK) return rc;
    kernel_timer_begin(st);
    kern<<<(unsigned)p.ctas, NT, smem, st>>>(p);
    kernel_timer_end(st);
    count_launch();
    NB_CUDA(cudaGetLastError());
    return NB_OK;
}

// The stream-K ranges of the packed positions; with `exponent`, also the
// call's fixed-point exponent (masses do not change within a step loop).
int launch_split(const SymParams &p, const ForceJob &j, const SymLayout &y, bool exponent) {
    NB_TRY_SYM(launch_pdl(sym_cost_kernel, (unsigned)cdiv(p.T * 32, 256), 256, 0, j.stream, p,
                          y.cost));
    NB_TRY_SYM(launch_pdl(sym_scan_kernel, 1, 1024, 0, j.stream, p, y.cost, y.prefix));
    NB_TRY_SYM(launch_pdl(sym_ranges_kernel, (unsigned)cdiv((p.ctas + 1) * 32, 128), 128, 0,
                          j.stream, p, y.prefix, y.lo));
    if (!exponent) return NB_OK;
    sym_exponent_kernel<<<(unsigned)std::min<int64_t>(cdiv(j.N, 4 * 256), 1024), 256, 0,
                          j.stream>>>(j.mass, j.N, j.eps, y.fx_exp, y.mmax_bits, y.arrivals,
                                      reinterpret_cast<ulonglong2 *>(y.acc_fx), 4 * p.Np);
    count_launch();
    NB_CUDA(cudaGetLastError());
    return NB_OK;
}

int launch_fold(const SymParams &p, const ForceJob &j, const int *perm, double *pot, double *vel,
                double kick) {
    const int64_t fold_blocks = std::min<int64_t>(cdiv(p.Np, 256), 64 * (int64_t)device_sm_count());
    sym_fold_kernel<<<(unsigned)fold_blocks, 256, 0, j.stream>>>(p, j.N, perm, j.G, j.acc, pot,
                                                                 vel, kick);
    count_launch();
    NB_CUDA(cudaGetLastError());
    return NB_OK;
}

template <int POL, int MODE>
int launch_pair_pot(const SymParams &p, bool pot, cudaStream_t st) {
    return pot ? launch_pair<POL, MODE, true>(p, st) : launch_pair<POL, MODE, false>(p, st);
}

template <int POL>
int launch_pair_mode(const SymParams &p, bool pot, cudaStream_t st) {
    switch (p.mode) {
        case 0: return launch_pair_pot<POL, 0>(p, pot, st);
        case 1: return launch_pair_pot<POL, 1>(p, pot, st);
        default: return launch_pair_pot<POL, 2>(p, pot, st);
    }
}

int launch_pair_pol(const SymParams &p, int precision, bool pot, cudaStream_t st) {
    switch (precision) {
        case NB_PREC_FP32: return launch_pair_mode<NB_PREC_FP32>(p, pot, st);
        case NB_PREC_KAHAN: return launch_pair_mode<NB_PREC_KAHAN>(p, pot, st);
        case NB_PREC_F64ACC: return launch_pair_mode<NB_PREC_F64ACC>(p, pot, st);
    }
    return fail(NB_ERR_INVALID, "unknown precision %d", precision);
}

SymParams params_of(const ForceJob &j, const SymLayout &y) {
    const SymSizes z = sym_sizes(j.L.Np);
    SymParams p;
    char *sb = j.ws + j.L.sortbuf;
    p.soa = reinterpret_cast<const float *>(j.ws + j.L.packA);
    p.Np = z.nb * kSymBlock;
    p.nb = z.nb;
    p.T = z.T;
    p.U = z.U;
    p.ctas = z.ctas;
    const float ef = (float)j.eps;
    p.eps2 = ef * ef;
    p.mode = j.adaptive ? 2 : (j.split ? 1 : 0);
    p.gamma = j.gamma;
    p.jbox = sort_tile_boxes(sb, j.L);
    p.wbox = sort_block_boxes(sb, j.L);
    p.acc_fx = y.acc_fx;
    p.fx_exp = y.fx_exp;
    p.lo = y.lo;
    p.status = reinterpret_cast<uint32_t *>(j.ws + j.L.status);
    return p;
}

// The pack of the current positions: in Hilbert order with its boxes, or (not
// adaptive) in particle order.
int pack_for(const SymParams &p, const ForceJob &j, bool reuse_order) {
    if (p.mode != 2)
        return launch_pack(j.pos, j.mass, j.N, j.L.Np,
                           reinterpret_cast<float *>(j.ws + j.L.packA), nullptr, 0, j.stream);
    char *sb = j.ws + j.L.sortbuf;
    return launch_sorted_pack(j.pos, j.mass, j.N, j.L.Np, reinterpret_cast<float *>(j.ws + j.L.packA),
                              nullptr, 0, sort_perm(sb, j.L), sort_keys(sb), sort_box6(sb, j.L),
                              sort_tile_boxes(sb, j.L), JSP, sort_block_boxes(sb, j.L), WS,
                              reuse_order, j.stream);
}

}  // namespace

SymSizes sym_sizes(int64_t Np) {
    SymSizes z{};
    z.nb = cdiv(Np, kSymBlock);
    z.T = z.nb * (z.nb + 1) / 2;
    z.U = z.T * US;
    z.ctas = std::min<int64_t>(CPS * (int64_t)device_sm_count(), z.U);
    z.fx_bytes = 8 * 8 * (size_t)(z.nb * kSymBlock);  // 4 components x 2 words per slot
    z.cost_bytes = align_up(4 * (size_t)z.T, 256) + align_up(8 * (size_t)(z.T + 1), 256) +
                   8 * (size_t)(z.ctas + 1);
    return z;
}

SymLayout sym_layout(char *ws, const WsLayout &L) {
    const SymSizes z = sym_sizes(L.Np);
    SymLayout y;
    char *c = ws + L.sym_cost, *head = ws + L.status;
    y.fx_exp = reinterpret_cast<int *>(head + kHeadSymExponent);
    y.mmax_bits = reinterpret_cast<unsigned long long *>(head + kHeadSymMaxMass);
    y.arrivals = reinterpret_cast<unsigned *>(head + kHeadSymArrivals);
    y.cost = reinterpret_cast<uint32_t *>(c);
    y.prefix = reinterpret_cast<unsigned long long *>(c + align_up(4 * (size_t)z.T, 256));
    y.lo = reinterpret_cast<int64_t *>(c + align_up(4 * (size_t)z.T, 256) +
                                       align_up(8 * (size_t)(z.T + 1), 256));
    y.acc_fx = reinterpret_cast<unsigned long long *>(ws + L.sym_fx);
    return y;
}

static int check_sym(const ForceJob &j) {
    if (j.eps <= 0.0) return fail(NB_ERR_UNSUPPORTED, "symmetric pairs need eps > 0");
    if (j.L.sym_fx_bytes == 0)
        return fail(NB_ERR_WORKSPACE, "workspace has no symmetric-pair buffers");
    return NB_OK;
}

int launch_force_sym(const ForceJob &j) {
    NB_TRY_SYM(check_sym(j));
    const SymLayout y = sym_layout(j.ws, j.L);
    const SymParams p = params_of(j, y);
    NB_TRY_SYM(pack_for(p, j, j.reuse_order));
    NB_TRY_SYM(launch_split(p, j, y, true));
    NB_TRY_SYM(launch_pair_pol(p, j.precision, j.pot != nullptr, j.stream));
    return launch_fold(p, j, p.mode == 2 ? sort_perm(j.ws + j.L.sortbuf, j.L) : nullptr, j.pot,
                       j.vel, j.kick);
}

int launch_step_sym(const ForceJob &j, double *vel, double dt, int64_t nsteps, bool acc_valid) {
    NB_TRY_SYM(check_sym(j));
    const SymLayout y = sym_layout(j.ws, j.L);
    const SymParams p = params_of(j, y);
    char *sb = j.ws + j.L.sortbuf;
    const bool sorted = p.mode == 2;
    const int *perm = sorted ? sort_perm(sb, j.L) : nullptr;
    const double half = 0.5 * dt;
    const int64_t e0 = acc_valid ? 1 : 0;  // evaluation 0 primes a(x)
    int64_t sorted_at = -1;
    bool opened = !acc_valid, packed = false;  // evaluation e's positions are there, are packed
    for (int64_t e = e0; e <= nsteps; ++e) {
        if (!opened)
            NB_TRY_SYM(launch_kick_drift_pack(const_cast<double *>(j.pos), vel, j.acc, j.mass, j.N,
                                              j.L.Np, dt, nullptr, nullptr, 0, j.stream));
        if (!packed) {
            const bool reuse = sorted_at >= 0 && e - sorted_at < kResortEvery;
            if (!reuse) sorted_at = e;
            NB_TRY_SYM(pack_for(p, j, reuse));
        }
        const bool last = e == nsteps;
        double *pot = last ? j.pot : nullptr;
        // the ranges follow the boxes; without them they are the same all along
        if (sorted || e == e0) NB_TRY_SYM(launch_split(p, j, y, e == e0));
        NB_TRY_SYM(launch_pair_pol(p, j.precision, pot != nullptr, j.stream));
        // the next evaluation keeps the order: its kick, drift and pack in the fold
        packed = !last && (!sorted || e + 1 - sorted_at < kResortEvery);
        opened = packed;
        auto next = sorted ? sym_fold_next_kernel<true> : sym_fold_next_kernel<false>;
        if (packed)
            NB_TRY_SYM(launch_pdl(next, (unsigned)(p.Np / 256), 256, 0, j.stream, p,
                                  j.N, perm, j.G, const_cast<double *>(j.pos), vel,
                                  e ? half : 0.0, half, dt,
                                  reinterpret_cast<float *>(j.ws + j.L.packA),
                                  sort_tile_boxes(sb, j.L), sort_block_boxes(sb, j.L)));
        else
            NB_TRY_SYM(launch_fold(p, j, perm, pot, e ? vel : nullptr, half));
    }
    return NB_OK;
}

}  // namespace nb
