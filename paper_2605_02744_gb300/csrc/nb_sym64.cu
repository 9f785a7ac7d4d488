// FP64 pairs with each unordered pair evaluated once, cut into one equal range
// of rotation steps per warp as in nb_wsym.cuh.
//
// FP64 runs at 1/64 of the FP32 rate on this part (two lanes a cycle per SM),
// so the pair term's 21 to 23 FP64 operations are all that counts: what feeds
// them (shuffles, integer atomics, loads) is free beside them, and a few warps
// per SM saturate the pipe.  What matters is that every SM gets the same number
// of pairs: the direct kernel gave each CTA 128 rows, i.e. 16 busy SMs at 2048
// particles and a second wave of five CTAs at 20001, and the earlier symmetric
// form had units of 2048 x 128 pairs.  A warp holds 64 i-slots (two per lane);
// a j-set is 32 particles, one per lane; a range may start and end at any
// rotation step.  Sums go into four-limb fixed-point totals (nb_fixed.cuh),
// exact whatever their order.
//
// The reciprocal square root is the hardware's seed (rsqrt.approx.ftz.f64)
// improved by one third-order Householder step, five FP64 operations, where
// the library call took about eight.  GB300, one evaluation with potentials:
// 16384 particles 10.78 ms (direct pairs) -> 5.42 ms, 2047: 1349 -> 99 us,
// 24577: 16.16 (earlier symmetric form) -> 12.26 ms.
#include <cuda_runtime.h>

#include <algorithm>

#include "nb_wsym.cuh"

namespace nb {

namespace {

using namespace wsym;

constexpr int K = 2;                 // i-slots per lane
constexpr int BW = 32 * K;           // slots per block
static_assert(BW >= kMinBlockSlots, "adds per total");
constexpr int WARPS = 8, NTHR = 32 * WARPS;
constexpr int JPB = K;               // j-sets of 32 per block

struct Params64 {
    const double *pos, *mass;  // [N][3], [N]
    int64_t N, Np, nb;
    int64_t per_warp, extra;   // rotation steps per warp; the first `extra` take one more
    double eps2;
    unsigned long long *fx;    // [4][4 limbs][Np]
    int *fxe;
    const unsigned long long *mx;  // max |m|, the bits of a double
    double scale;              // bound of every partial and total / max|m|
    uint32_t *status;
};

// 1 / sqrt(x), x >= 0 and not denormal: the seed y has a relative error below
// 2^-19, e = 1 - x y^2 and y (1 + e / 2 + 3 e^2 / 8) leaves 5 e^3 / 16, below
// 2^-54, and the rounding of the last operation.  An infinite x keeps the
// seed's 0, a NaN its NaN.
__device__ __forceinline__ double rsqrt64(double x) {
    double y;
    asm("rsqrt.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(x));
    const double e = fma(-(x * y), y, 1.0);
    const double z = fma(fma(0.375, e, 0.5), y * e, y);
    return __double2hiint(x) >= 0x7ff00000 ? y : z;
}

struct ISet {
    double x[K], y[K], z[K], m[K];
    double ax[K], ay[K], az[K], ph[K];
};

template <bool SYM, bool SELF, bool POT>
__device__ __forceinline__ void step(ISet &S, double eps2, double jx, double jy, double jz,
                                     double jm, double (&b)[4], int self_k) {
#pragma unroll
    for (int k = 0; k < K; ++k) {
        const double mj = (SELF && k == self_k) ? 0.0 : jm;
        const double dx = jx - S.x[k], dy = jy - S.y[k], dz = jz - S.z[k];
        const double r2 = fma(dx, dx, fma(dy, dy, fma(dz, dz, eps2)));
        const double r = rsqrt64(r2);
        const double r3 = r * r * r;
        const double sj = mj * r3;
        S.ax[k] = fma(sj, dx, S.ax[k]);
        S.ay[k] = fma(sj, dy, S.ay[k]);
        S.az[k] = fma(sj, dz, S.az[k]);
        if (POT) S.ph[k] = fma(mj, r, S.ph[k]);
        if (SYM) {
            const double si = S.m[k] * r3;
            b[0] = fma(-si, dx, b[0]);
            b[1] = fma(-si, dy, b[1]);
            b[2] = fma(-si, dz, b[2]);
            if (POT) b[3] = fma(S.m[k], r, b[3]);
        }
    }
}

// n rotation steps of one j-set; the sums end one lane behind, as in
// wsym::rotate.
template <bool SYM, bool POT>
__device__ __forceinline__ void rotate64(ISet &S, double eps2, const double (&j)[4],
                                         double (&b)[4], int n, int self_k) {
    const int src = (threadIdx.x + 1) & 31;
    double J[4] = {j[0], j[1], j[2], j[3]};
#pragma unroll
    for (int e = 0; e < 4; ++e) b[e] = 0.0;
    auto one = [&](auto self) {
        double Jn[4];
#pragma unroll
        for (int a = 0; a < 4; ++a) Jn[a] = __shfl_sync(0xffffffffu, J[a], src);
        if (SYM) {
#pragma unroll
            for (int e = 0; e < (POT ? 4 : 3); ++e) b[e] = __shfl_sync(0xffffffffu, b[e], src);
        }
        step<SYM, decltype(self)::value, POT>(S, eps2, J[0], J[1], J[2], J[3], b, self_k);
#pragma unroll
        for (int a = 0; a < 4; ++a) J[a] = Jn[a];
    };
    int st = 0;
    if (!SYM && self_k >= 0) {
        one(std::true_type{});
        st = 1;
    }
#pragma unroll 2
    for (; st < n; ++st) one(std::false_type{});
}

__device__ __forceinline__ void load64(const Params64 &p, int s, double (&j)[4]) {
    if (s < p.N) {
        j[0] = p.pos[3 * (int64_t)s];
        j[1] = p.pos[3 * (int64_t)s + 1];
        j[2] = p.pos[3 * (int64_t)s + 2];
        j[3] = p.mass[s];
    } else {
        j[0] = j[1] = j[2] = j[3] = 0.0;  // padding: zero mass at the origin
    }
}

template <bool POT>
__global__ void __launch_bounds__(NTHR) sym64_kernel(const Params64 p) {
    __shared__ int sF;
    const int tid = threadIdx.x, w = tid >> 5, l = tid & 31;
    const int64_t gw = (int64_t)blockIdx.x * WARPS + w;
    int64_t u = gw * p.per_warp + (gw < p.extra ? gw : p.extra);
    const int64_t u_end = u + p.per_warp + (gw < p.extra ? 1 : 0);
    int I = 0, jb = 0;
    if (u < u_end) {
        int J;
        item_of(u / (32 * JPB), p.nb, I, J);
        jb = J * BW + (int)(u % (32 * JPB)) / 32 * 32;
    }
    dev::grid_wait();
    if (tid == 0) {
        sF = fx::limb_exponent_for(p.scale * __longlong_as_double((long long)__ldcg(p.mx)));
        if (blockIdx.x == 0) *p.fxe = sF;
    }
    __syncthreads();
    const int F = sF;
    const int nslots = (int)(p.nb * BW);
    uint32_t bad = 0;
    auto add = [&](int e, int slot, double v) {
        int q;
        long long t[3];
        const bool ok = fx::split_limbs(v, F, q, t);
        if (slot >= p.N) return;
        unsigned long long *wd = p.fx + (int64_t)(fx::kLimbs * e + q) * p.Np + slot;
        if (!ok) {
            bad = 1;
            poison(wd + (fx::kLimbs - 1) * p.Np);  // q is 0
        }
#pragma unroll
        for (int k = 0; k < 3; ++k)
            if (t[k]) atomicAdd(wd + k * p.Np, (unsigned long long)t[k]);
    };
    ISet S;
    bool open = false;
    while (u < u_end) {
        const int s0 = (int)u & 31;
        const int n = u_end - u < 32 - s0 ? (int)(u_end - u) : 32 - s0;
        if (!open) {
#pragma unroll
            for (int k = 0; k < K; ++k) {
                double v[4];
                load64(p, I * BW + 32 * k + l, v);
                S.x[k] = v[0];
                S.y[k] = v[1];
                S.z[k] = v[2];
                S.m[k] = v[3];
                S.ax[k] = S.ay[k] = S.az[k] = S.ph[k] = 0.0;
            }
            open = true;
        }
        double j[4], b[4];
        load64(p, jb + ((l + s0) & 31), j);
        u += n;
        if (jb >= (I + 1) * BW) {
            rotate64<true, POT>(S, p.eps2, j, b, n, -1);
            const int js = jb + ((l + s0 + n - 1) & 31);
#pragma unroll
            for (int e = 0; e < (POT ? 4 : 3); ++e) add(e, js, b[e]);
        } else {
            rotate64<false, POT>(S, p.eps2, j, b, n, s0 == 0 ? (jb - I * BW) / 32 : -1);
        }
        jb += 32;
        if (u >= u_end || jb >= nslots) {  // end of the warp's segment of row I
#pragma unroll
            for (int k = 0; k < K; ++k) {
                const double v[4] = {S.ax[k], S.ay[k], S.az[k], S.ph[k]};
#pragma unroll
                for (int e = 0; e < (POT ? 4 : 3); ++e) add(e, I * BW + 32 * k + l, v[e]);
            }
            ++I;
            jb = I * BW;
            open = false;
        }
    }
    if (bad) dev::set_status(p.status, kStatusNonFinite);
}

// The largest |m|, after an optional kick and drift (v += kick a; x += drift v),
// and cleared totals.
__global__ void __launch_bounds__(128) sym64_open_kernel(double *pos, double *vel,
                                                         const double *acc, const double *mass,
                                                         int64_t N, double kick, double drift,
                                                         unsigned long long *mx,
                                                         unsigned long long *fx, int64_t Np,
                                                         int nc) {
    const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    dev::grid_trigger();
    dev::grid_wait();
    if (clear_totals(fx, N, N, Np, nc)) return;
    unsigned long long am = 0ull;  // non-negative doubles order like their bits
    if (i < N) {
        if (vel) {
#pragma unroll
            for (int c = 0; c < 3; ++c) {
                const double v = vel[3 * i + c] + kick * acc[3 * i + c];
                vel[3 * i + c] = v;
                pos[3 * i + c] += drift * v;
            }
        }
        am = (unsigned long long)__double_as_longlong(fabs(mass[i]));
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        const unsigned long long v = __shfl_xor_sync(0xffffffffu, am, o);
        am = v > am ? v : am;
    }
    if ((threadIdx.x & 31) == 0 && am) atomicMax(mx, am);
}

// The totals of every particle, as wsym_fold_kernel; NEXT: also the next
// step's opening kick and drift.
template <bool NEXT>
__global__ void __launch_bounds__(128) sym64_fold_kernel(const Params64 p, double G, double *acc,
                                                         double *pot, double *pos, double *vel,
                                                         double kick, double next_kick,
                                                         double drift,
                                                         unsigned long long *mx) {
    const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    dev::grid_trigger();
    dev::grid_wait();
    if (!NEXT && i == 0) *mx = 0ull;  // for the next call
    if (i >= p.N) return;
    Params t{};
    t.fx = p.fx;
    t.Np = p.Np;
    const int F = *p.fxe;
    bool ok = true;
#pragma unroll
    for (int c = 0; c < 3; ++c) {
        const double a = G * take_fixed(t, c, i, F);
        ok = ok && isfinite(a);
        if (!NEXT) acc[3 * i + c] = a;
        if (vel) {
            double v = vel[3 * i + c] + kick * a;
            if (NEXT) {
                v = v + next_kick * a;
                pos[3 * i + c] += drift * v;
            }
            vel[3 * i + c] = v;
        }
    }
    if (!NEXT && pot) {
        const double gp = -G * take_fixed(t, 3, i, F);
        pot[i] = gp;
        ok = ok && isfinite(gp);
    }
    if (!ok) dev::set_status(p.status, kStatusNonFinite);
}

struct Run64 {
    const ForceJob &j;
    Params64 p{};
    unsigned long long *mx;

    explicit Run64(const ForceJob &job) : j(job) {
        mx = reinterpret_cast<unsigned long long *>(j.ws + j.L.status + kHeadMaxMass64);
        p.pos = j.pos;
        p.mass = j.mass;
        p.N = j.N;
        p.Np = j.L.Np;
        p.eps2 = j.eps * j.eps;
        p.fx = reinterpret_cast<unsigned long long *>(j.ws + j.L.wsym_fx);
        p.fxe = reinterpret_cast<int *>(j.ws + j.L.status + kHeadExponents);
        p.mx = mx;
        p.status = reinterpret_cast<uint32_t *>(j.ws + j.L.status);
        // as params_of in nb_wsym.cu
        p.scale = 1.02 * (double)j.N * std::max(0.3849002 / (j.eps * j.eps), 1.0 / j.eps);
        p.nb = cdiv(j.N, BW);
    }
    int open(double *vel, double kick, double drift) {
        const int nc = j.pot ? 4 : 3;
        return launch_pdl(sym64_open_kernel, pack_blocks(j.N, j.N, nc), 128, 0, j.stream,
                          const_cast<double *>(j.pos), vel, j.acc, j.mass, j.N, kick, drift, mx, p.fx,
                          p.Np, nc);
    }
    int pairs(bool pot) {
        auto kern = pot ? sym64_kernel<true> : sym64_kernel<false>;
        const int64_t steps = p.nb * (p.nb + 1) / 2 * JPB * 32;
        static const int occ = std::min(
            2, occupancy(reinterpret_cast<const void *>(sym64_kernel<true>), NTHR, 0));
        const int64_t ctas = std::min<int64_t>(occ * (int64_t)device_sm_count(), cdiv(steps, WARPS));
        p.per_warp = steps / (ctas * WARPS);
        p.extra = steps % (ctas * WARPS);
        return launch_pdl(kern, (unsigned)ctas, NTHR, 0, j.stream, p);
    }
    int fold(double *pot, bool next, double *vel, double kick, double next_kick, double drift) {
        auto k = next ? sym64_fold_kernel<true> : sym64_fold_kernel<false>;
        return launch_pdl(k, (unsigned)cdiv(j.N, 128), 128, 0, j.stream, p, j.G, j.acc, pot,
                          const_cast<double *>(j.pos), vel, kick, next_kick, drift, mx);
    }
};

}  // namespace

int launch_force_sym64(const ForceJob &j) {
    Run64 r(j);
    int rc = r.open(nullptr, 0.0, 0.0);
    if (rc || (rc = r.pairs(j.pot != nullptr))) return rc;
    return r.fold(j.pot, false, j.vel, j.kick, 0.0, 0.0);
}

int launch_step_sym64(const ForceJob &j, double *vel, double dt, int64_t nsteps, bool acc_valid) {
    Run64 r(j);
    const double half = 0.5 * dt;
    int rc = r.open(acc_valid ? vel : nullptr, half, dt);
    if (rc) return rc;
    // evaluation e = 0 is the priming one when a(x) is not known yet
    for (int64_t e = acc_valid ? 1 : 0; e <= nsteps; ++e) {
        const bool next = e < nsteps;
        double *pot = next ? nullptr : j.pot;
        if ((rc = r.pairs(pot != nullptr))) return rc;
        if ((rc = r.fold(pot, next, nsteps ? vel : nullptr, e ? half : 0.0, half, dt))) return rc;
    }
    return NB_OK;
}

}  // namespace nb
