// Forces of one small system (every ordered pair), one kernel per evaluation.
//
// Below a few thousand particles the evaluation is a handful of microseconds
// of arithmetic, and what costs is everything around it: the tiled direct
// kernel spent its time (F64ACC step: 17.6 us at 1024 particles, 34.6 us at
// 4095) on partial records, arrival counters, a fixup chain and a second
// kernel for the kick, drift and pack.  Here a CTA owns a few whole rows, so
// its sums never leave it, and inside an nb_step loop the thread that
// finishes a particle's acceleration also does its closing kick and the next
// step's kick, drift and pack (into the other of two packed buffers, because
// other CTAs still read this one): one launch a step, no scratch in memory.
// Measured the same way: 3.9 us at 1024, 16.2 us at 4095.  What bounds it now
// is the FP32 pipe from about 2000 particles (60 % busy at 4095), and below
// that the launch and the dependent loads of a step (2.8 us at 64).
//
// The warps split the j-particles: each takes every fourth set of 64 (two per
// lane, packed f32x2, read from L1 / L2), against four rows at a time held
// broadcast in registers (dev::pair2: 18 packed FP32 operations per two hi/lo
// pairs, 19 with the potential).  The lanes' sums of four rows are combined
// with a reduce-scatter over the warp (16 shuffles for 16 values), the warps'
// sums in shared memory in FP64 (F64ACC) or as compensated float pairs.  So a
// sum of plain FP32 adds covers N / 256 terms per lane and the tree over 64 of
// them, and the rest is of the policy's own kind.
#include <cuda_runtime.h>

#include <algorithm>

#include "nb_device.cuh"
#include "nb_fpconv.cuh"
#include "nb_internal.h"

namespace nb {

using dev::f2;
using dev::pair2;

namespace {

// Four CTAs of 4 warps per SM rather than two of 8: the same time for one
// system (4095: 16.2 / 15.4 us a step, 2047: 6.3 / 6.6), and several systems
// stepped on several streams overlap better (12.4 / 13.5 us a step at 4095).
constexpr int NW = 4, NT = 32 * NW, CPS = 4;
constexpr int kMaxRows = 16;        // rows per CTA at most

// The packed buffers here are tiled: 64 particles' x.hi y.hi z.hi m x.lo y.lo
// z.lo, 64 floats each, so that a j-set's loads share one address (with the
// [7][Np] arrays of the other kernels a third of this kernel's instructions
// were address arithmetic).
constexpr int TILE = 7 * 64;
__host__ __device__ __forceinline__ int64_t at(int a, int64_t i) {
    return (i >> 6) * TILE + a * 64 + (i & 63);
}

struct RowParams {
    const float *soa;   // packed tiles of this evaluation's positions
    float *soa_next;    // NEXT: the buffer of the next one
    int64_t N, Np;
    float eps2;
    double G;
    double *acc, *pot, *pos, *vel;
    double kick, next_kick, drift;
    uint32_t *status;
};

// TwoSum (Knuth): (s, c) + x without losing the rounding error.
__device__ __forceinline__ void two_add(float2 &t, float x) {
    const float s = __fadd_rn(t.x, x);
    const float z = __fsub_rn(s, t.x);
    t.y = __fadd_rn(t.y, __fadd_rn(__fsub_rn(t.x, __fsub_rn(s, z)), __fsub_rn(x, z)));
    t.x = s;
}

// Sums each v[i] over the warp by halving the values a lane carries with every
// exchange; lane l ends with the sum of value l / (32 / NV).
template <int NV>
__device__ __forceinline__ float reduce_lanes(float (&v)[NV]) {
    const int l = threadIdx.x & 31;
    int o = 16;
#pragma unroll
    for (int h = NV / 2; h >= 1; h >>= 1, o >>= 1) {
        const bool up = l & o;
#pragma unroll
        for (int i = 0; i < h; ++i) {
            const float keep = up ? v[i + h] : v[i], give = up ? v[i] : v[i + h];
            v[i] = keep + __shfl_xor_sync(0xffffffffu, give, o);
        }
    }
#pragma unroll
    for (; o >= 1; o >>= 1) v[0] += __shfl_xor_sync(0xffffffffu, v[0], o);
    return v[0];
}

// Rows g .. g + RG - 1 of the CTA against every j-set of this warp; the sums
// go to part[w].
template <int RG, bool SPLIT, bool POT>
__device__ __forceinline__ void row_group(const RowParams &p, int r0, int nr, int g,
                                          const float (&rows)[6][kMaxRows],
                                          float (&part)[kMaxRows * 4]) {
    const int w = threadIdx.x >> 5, l = threadIdx.x & 31;
    const int sets = (int)((p.N + 63) / 64);
    const float2 e2 = f2(p.eps2, p.eps2);
    float2 nx[RG], ny[RG], nz[RG], nxl[RG], nyl[RG], nzl[RG];
    float2 ax[RG], ay[RG], az[RG], ph[RG];
    int kr[RG];
#pragma unroll
    for (int k = 0; k < RG; ++k) {
        const int r = g + k < nr ? g + k : nr - 1;  // past the rows: the last one again
        nx[k] = f2(rows[0][r], rows[0][r]);
        ny[k] = f2(rows[1][r], rows[1][r]);
        nz[k] = f2(rows[2][r], rows[2][r]);
        nxl[k] = f2(rows[3][r], rows[3][r]);
        nyl[k] = f2(rows[4][r], rows[4][r]);
        nzl[k] = f2(rows[5][r], rows[5][r]);
        kr[k] = r0 + r;
        ax[k] = ay[k] = az[k] = ph[k] = f2(0.f, 0.f);
    }
    const float *jp = p.soa + 2 * l;
#pragma unroll 1
    for (int s = w; s < sets; s += NW) {
        const int j = 64 * s + 2 * l;
        float2 v[7];
#pragma unroll
        for (int a = 0; a < (SPLIT ? 7 : 4); ++a)
            v[a] = *reinterpret_cast<const float2 *>(jp + s * TILE + 64 * a);
        if (!SPLIT) v[4] = v[5] = v[6] = f2(0.f, 0.f);
        if (64 * s < r0 + nr && 64 * s + 64 > r0)  // some of the rows themselves
            pair2<RG, false, SPLIT, true>(v[0], v[1], v[2], v[4], v[5], v[6], v[3], e2, nx, ny, nz,
                                          nxl, nyl, nzl, ax, ay, az, ph, kr, j);
        else
            pair2<RG, false, SPLIT, false>(v[0], v[1], v[2], v[4], v[5], v[6], v[3], e2, nx, ny,
                                           nz, nxl, nyl, nzl, ax, ay, az, ph);
    }
    float v[4 * RG];
#pragma unroll
    for (int k = 0; k < RG; ++k) {
        v[4 * k] = ax[k].x + ax[k].y;
        v[4 * k + 1] = ay[k].x + ay[k].y;
        v[4 * k + 2] = az[k].x + az[k].y;
        v[4 * k + 3] = POT ? ph[k].x + ph[k].y : 0.f;
    }
    const float sum = reduce_lanes<4 * RG>(v);
    constexpr int LPV = 8 / RG;  // lanes per value
    if (l % LPV == 0 && 4 * g + l / LPV < 4 * nr) part[4 * g + l / LPV] = sum;
}

// F64: the warps' sums are added in FP64 (F64ACC), else as a compensated float
// pair.
template <bool SPLIT, bool POT, bool NEXT, bool F64>
__global__ void __launch_bounds__(NT, CPS) row_kernel(const RowParams p) {
    __shared__ float rows[6][kMaxRows];
    __shared__ float part[NW][kMaxRows * 4];  // [warp][row][component]
    const int tid = threadIdx.x, w = tid >> 5;
    // whole pairs of rows per CTA: row groups are 4 or 2 rows
    const int64_t half = (p.N + 1) / 2;
    const int r0 = 2 * (int)(half * blockIdx.x / gridDim.x);
    const int r1 = 2 * (int)(half * (blockIdx.x + 1) / gridDim.x);
    const int nr = (r1 < (int)p.N ? r1 : (int)p.N) - r0;
    dev::grid_trigger();
    dev::grid_wait();
    for (int v = tid; v < 6 * nr; v += NT) {
        const int a = v / nr, r = v % nr;
        rows[a][r] = -p.soa[at(a < 3 ? a : a + 1, r0 + r)];
    }
    __syncthreads();
    int g = 0;
#pragma unroll 1
    for (; g + 2 < nr; g += 4) row_group<4, SPLIT, POT>(p, r0, nr, g, rows, part[w]);
    if (g < nr) row_group<2, SPLIT, POT>(p, r0, nr, g, rows, part[w]);
    __syncthreads();
    for (int v = tid; v < 4 * nr; v += NT) {
        const int c = v & 3;
        if (c == 3 && !POT) continue;
        const int64_t i = r0 + (v >> 2);
        double sum;
        if (F64) {
            static_assert(NW == 4, "a tree over the warps");
            sum = (fpconv::f2d(part[0][v]) + fpconv::f2d(part[1][v])) +
                  (fpconv::f2d(part[2][v]) + fpconv::f2d(part[3][v]));
        } else {
            float2 t = f2(0.f, 0.f);
#pragma unroll
            for (int w2 = 0; w2 < NW; ++w2) two_add(t, part[w2][v]);
            sum = fpconv::f2d(t.x) + fpconv::f2d(t.y);
        }
        const double a = p.G * sum;
        if (!fpconv::finite_d(a)) dev::set_status(p.status, kStatusNonFinite);
        if (c == 3) {
            p.pot[i] = -a;
            continue;
        }
        if (!NEXT) p.acc[3 * i + c] = a;
        if (p.vel) {
            double u = p.vel[3 * i + c] + p.kick * a;
            if (NEXT) {
                u = u + p.next_kick * a;
                const double x = p.pos[3 * i + c] + p.drift * u;
                p.pos[3 * i + c] = x;
                const float h = fpconv::d2f(x);
                p.soa_next[at(c, i)] = h;
                p.soa_next[at(4 + c, i)] = fpconv::d2f(x - fpconv::f2d(h));
            }
            p.vel[3 * i + c] = u;
        }
    }
}

template <bool SPLIT, bool F64>
int launch_row(const RowParams &p, bool next, cudaStream_t st) {
    const int64_t ctas = std::min<int64_t>(CPS * device_sm_count(), (p.N + 1) / 2);
    auto k = next ? row_kernel<SPLIT, false, true, F64>
                  : (p.pot ? row_kernel<SPLIT, true, false, F64>
                           : row_kernel<SPLIT, false, false, F64>);
    return launch_pdl(k, (unsigned)ctas, NT, 0, st, p);
}

// Both packed buffers: positions after an optional kick and drift (v += kick
// a; x += drift v) into the first, the masses (which do not change) and the
// zero padding into both.
__global__ void __launch_bounds__(128) row_pack_kernel(double *pos,
                                                       double *vel,
                                                       const double *acc,
                                                       const double *mass, int64_t N,
                                                       int64_t Np, double kick, double drift,
                                                       float *soa,
                                                       float *soa2) {
    const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;  // < Np: whole blocks
    float hi[3] = {0.f, 0.f, 0.f}, lo[3] = {0.f, 0.f, 0.f}, m = 0.f;
    dev::grid_trigger();
    dev::grid_wait();
    if (i < N) {
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            double x = pos[3 * i + c];
            if (vel) {
                const double v = vel[3 * i + c] + kick * acc[3 * i + c];
                x = x + drift * v;
                vel[3 * i + c] = v;
                pos[3 * i + c] = x;
            }
            hi[c] = fpconv::d2f(x);
            lo[c] = fpconv::d2f(x - fpconv::f2d(hi[c]));
        }
        m = fpconv::d2f(mass[i]);
    }
#pragma unroll
    for (int c = 0; c < 3; ++c) {
        soa[at(c, i)] = hi[c];
        soa[at(4 + c, i)] = lo[c];
        if (soa2 && i >= N) soa2[at(c, i)] = soa2[at(4 + c, i)] = 0.f;
    }
    soa[at(3, i)] = m;
    if (soa2) soa2[at(3, i)] = m;
}

int pack_rows(const ForceJob &j, double *vel, double kick, double drift, bool both) {
    return launch_pdl(row_pack_kernel, (unsigned)(j.L.Np / 128), 128, 0, j.stream,
                      const_cast<double *>(j.pos), vel, j.acc, j.mass, j.N, j.L.Np, kick, drift,
                      reinterpret_cast<float *>(j.ws + j.L.packA),
                      both ? reinterpret_cast<float *>(j.ws + j.L.cot64) : nullptr);
}

RowParams params_of(const ForceJob &j) {
    RowParams p{};
    p.soa = reinterpret_cast<const float *>(j.ws + j.L.packA);
    p.N = j.N;
    p.Np = j.L.Np;
    const float ef = (float)j.eps;
    p.eps2 = ef * ef;
    p.G = j.G;
    p.acc = j.acc;
    p.pot = j.pot;
    p.pos = const_cast<double *>(j.pos);
    p.status = reinterpret_cast<uint32_t *>(j.ws + j.L.status);
    return p;
}

int launch_rows(const ForceJob &j, const RowParams &p, bool next) {
    if (j.precision == NB_PREC_F64ACC)
        return j.split ? launch_row<true, true>(p, next, j.stream)
                       : launch_row<false, true>(p, next, j.stream);
    return j.split ? launch_row<true, false>(p, next, j.stream)
                   : launch_row<false, false>(p, next, j.stream);
}

}  // namespace

bool row_fits(int64_t N) { return cdiv(N, 2 * CPS * device_sm_count()) * 2 <= kMaxRows; }

int launch_force_row(const ForceJob &j) {
    RowParams p = params_of(j);
    p.vel = j.vel;
    p.kick = j.kick;
    const int rc = pack_rows(j, nullptr, 0.0, 0.0, false);
    return rc ? rc : launch_rows(j, p, false);
}

int launch_step_row(const ForceJob &j, double *vel, double dt, int64_t nsteps, bool acc_valid) {
    const double half = 0.5 * dt;
    int rc = pack_rows(j, acc_valid ? vel : nullptr, half, dt, true);
    if (rc) return rc;
    RowParams p = params_of(j);
    p.next_kick = half;
    p.drift = dt;
    float *buf[2] = {reinterpret_cast<float *>(j.ws + j.L.packA),
                     reinterpret_cast<float *>(j.ws + j.L.cot64)};
    int cur = 0;
    // evaluation e = 0 is the priming one when a(x) is not known yet
    for (int64_t e = acc_valid ? 1 : 0; e <= nsteps; ++e, cur ^= 1) {
        const bool next = e < nsteps;
        p.soa = buf[cur];
        p.soa_next = buf[cur ^ 1];
        p.pot = next ? nullptr : j.pot;
        p.vel = nsteps ? vel : nullptr;
        p.kick = e ? half : 0.0;
        if ((rc = launch_rows(j, p, next))) return rc;
    }
    return NB_OK;
}

}  // namespace nb
