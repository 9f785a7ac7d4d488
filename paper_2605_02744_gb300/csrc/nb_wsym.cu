// Forces of one system by the warp-granular symmetric-pair engine
// (nb_wsym.cuh), with one displacement form for every pair: single floats or
// hi/lo pairs.  Three kernels per evaluation -- pack (with the largest mass),
// pairs, fold -- and two per step inside an nb_step loop, where the fold of
// one step also does the next step's kick, drift and pack.
#include <cuda_runtime.h>

#include <algorithm>

#include "nb_wsym.cuh"

namespace nb {

using namespace wsym;

namespace {

// a_i = sum m_j r^-3 d and phi: 18 FP32 operations per unordered pair, 24
// with the hi/lo displacement (16 / 22 without the potential).
template <bool IPAIR_, int K_, int WARPS_, bool SPLIT, bool POT>
struct ForcePh {
    static constexpr bool IPAIR = IPAIR_;
    static constexpr int K = K_, WARPS = WARPS_, NJ = SPLIT ? 7 : 4, NC = POT ? 4 : 3;
    static constexpr int GROUPS = POT ? 2 : 1;
    struct S {
        float2 nx[K], ny[K], nz[K], m[K];
        LoT<IPAIR> nxl[K], nyl[K], nzl[K];
        float2 a[K][NC];
    };
    static __device__ __forceinline__ constexpr int group(int e) { return e < 3 ? 0 : 1; }
    static __device__ __forceinline__ constexpr bool jneg(int e) { return e < 3; }
    static __device__ __forceinline__ int bound(const Params &p, const Maxima &x, int g) {
        return p.sexp[g] + x.m;
    }
    // groups: accelerations, potential
    static __device__ __forceinline__ int shift(const Scales &z, int g) {
        return g == 0 ? z.m - 2 * z.x : z.m - z.x;
    }
    static __device__ __forceinline__ constexpr int factor(int a) { return a == 3 ? kFm : kFx; }
    static __device__ __forceinline__ const float *plane(const Params &p, int a) {
        return p.soa + a * p.Np;
    }
    static __device__ __forceinline__ void set_i(S &s, int k, const float2 (&v)[NJ]) {
        s.nx[k] = neg(v[0]);
        s.ny[k] = neg(v[1]);
        s.nz[k] = neg(v[2]);
        s.m[k] = v[3];
        if constexpr (SPLIT) {
            s.nxl[k] = lo_of<IPAIR>(neg(v[4]));
            s.nyl[k] = lo_of<IPAIR>(neg(v[5]));
            s.nzl[k] = lo_of<IPAIR>(neg(v[6]));
        }
    }
    template <bool SYM, bool SELF>
    static __device__ __forceinline__ void step(S &s, const float2 e2, const float2 (&J)[NJ],
                                                float2 (&T)[NC], int self_h) {
#pragma unroll
        for (int k = 0; k < K; ++k) {
            float2 dx = add2(J[0], s.nx[k]);
            float2 dy = add2(J[1], s.ny[k]);
            float2 dz = add2(J[2], s.nz[k]);
            if constexpr (SPLIT) {
                dx = add2(dx, add2(J[4], lo2(s.nxl[k])));
                dy = add2(dy, add2(J[5], lo2(s.nyl[k])));
                dz = add2(dz, add2(J[6], lo2(s.nzl[k])));
            }
            float2 r2 = fma2(dx, dx, e2);
            r2 = fma2(dy, dy, r2);
            r2 = fma2(dz, dz, r2);
            float2 r = f2(rsqrt_approx(r2.x), rsqrt_approx(r2.y));
            if (SELF) r = mask_self<IPAIR>(r, k, self_h);
            const float2 r3 = mul2(mul2(r, r), r);
            const float2 sj = mul2(J[3], r3);
            s.a[k][0] = fma2(sj, dx, s.a[k][0]);
            s.a[k][1] = fma2(sj, dy, s.a[k][1]);
            s.a[k][2] = fma2(sj, dz, s.a[k][2]);
            if constexpr (POT) s.a[k][3] = fma2(J[3], r, s.a[k][3]);
            if (SYM) {
                const float2 si = mul2(s.m[k], r3);
                T[0] = k ? fma2(si, dx, T[0]) : mul2(si, dx);
                T[1] = k ? fma2(si, dy, T[1]) : mul2(si, dy);
                T[2] = k ? fma2(si, dz, T[2]) : mul2(si, dz);
                if constexpr (POT) T[3] = k ? fma2(s.m[k], r, T[3]) : mul2(s.m[k], r);
            }
        }
    }
};

// Pack of the positions and masses after an optional kick and drift
// (v += kick a; x += drift v), the largest |m| and |x|, and cleared totals (nc
// components).
__global__ void __launch_bounds__(128) wsym_pack_kernel(double *pos,
                                                        double *vel,
                                                        const double *acc,
                                                        const double *mass, int64_t N,
                                                        int64_t Np, double kick, double drift,
                                                        float *soa, unsigned *mx,
                                                        unsigned long long *fx, int nc) {
    const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;  // < Np: whole blocks
    float hi[3] = {0.f, 0.f, 0.f}, lo[3] = {0.f, 0.f, 0.f}, m = 0.f, am = 0.f, ax = 0.f;
    dev::grid_trigger();
    dev::grid_wait();
    if (clear_totals(fx, Np, N, Np, nc)) return;
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
            hi[c] = __double2float_rn(x);
            lo[c] = __double2float_rn(x - (double)hi[c]);
        }
        const double md = mass[i];
        m = __double2float_rn(md);
        am = __double2float_ru(fabs(md));
        ax = fmaxf(fabsf(hi[0]), fmaxf(fabsf(hi[1]), fabsf(hi[2])));
    } else {
        hi[0] = kPadX;
    }
    store_packed(soa, Np, i, hi, lo, m);
    warp_max(mx + kMaxM, am);
    warp_max(mx + kMaxX, ax);
}

// The totals of every particle: read and zeroed, x G, stored, with an optional
// closing kick; NEXT: also the next step's opening kick, drift and pack (its
// masses are already packed), and no store of the acceleration, which the
// next step's fold replaces before anything reads it.
template <bool NEXT>
__global__ void __launch_bounds__(128) wsym_fold_kernel(const Params p, double G,
                                                        double *acc,
                                                        double *pot,
                                                        double *pos,
                                                        double *vel, double kick,
                                                        double next_kick, double drift,
                                                        float *soa, unsigned *mx) {
    const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    dev::grid_trigger();
    dev::grid_wait();
    if (!NEXT && i == 0) mx[kMaxM] = mx[kMaxX] = 0u;  // for the next call
    if (i >= p.N) return;
    const int F = *p.fxe;
    double x0[3], v0[3];
    if (vel) {
#pragma unroll
        for (int c = 0; c < 3; ++c) v0[c] = vel[3 * i + c];
    }
    if (NEXT) {
#pragma unroll
        for (int c = 0; c < 3; ++c) x0[c] = pos[3 * i + c];
    }
    double a[3];
    bool ok = true;
#pragma unroll
    for (int c = 0; c < 3; ++c) {
        a[c] = G * take_fixed(p, c, i, F);
        ok = ok && isfinite(a[c]);
        if (!NEXT) acc[3 * i + c] = a[c];
        if (vel) {
            double v = v0[c] + kick * a[c];
            if (NEXT) {
                v = v + next_kick * a[c];
                const double x = x0[c] + drift * v;
                pos[3 * i + c] = x;
                const float h = __double2float_rn(x);
                soa[c * p.Np + i] = h;
                soa[(4 + c) * p.Np + i] = __double2float_rn(x - (double)h);
            }
            vel[3 * i + c] = v;
        }
    }
    if (!NEXT && pot) {
        const double gp = -G * take_fixed(p, 3, i, p.fxe[1]);
        pot[i] = gp;
        ok = ok && isfinite(gp);
    }
    if (!ok) dev::set_status(p.status, kStatusNonFinite);
}

unsigned *maxima(const ForceJob &j) {
    return reinterpret_cast<unsigned *>(j.ws + j.L.status + kHeadMaxima);
}

Params params_of(const ForceJob &j) {
    Params p{};
    p.soa = reinterpret_cast<const float *>(j.ws + j.L.packA);
    p.Np = j.L.Np;
    p.N = j.N;
    p.eps = (float)j.eps;
    p.keep = j.precision != NB_PREC_FP32;
    p.fx = reinterpret_cast<unsigned long long *>(j.ws + j.L.wsym_fx);
    p.fxe = reinterpret_cast<int *>(j.ws + j.L.status + kHeadExponents);
    p.mx = maxima(j);
    p.status = reinterpret_cast<uint32_t *>(j.ws + j.L.status);
    // every partial and total: N max|m| times the largest |d| (|d|^2 +
    // eps^2)^-3/2 (0.385 / eps^2) and (|d|^2 + eps^2)^-1/2 (1 / eps), x 1.02
    // for the rounding of the FP32 partial sums
    p.set_scale(0, 1.02 * (double)j.N * 0.3849002 / (j.eps * j.eps));
    p.set_scale(1, 1.02 * (double)j.N / j.eps);
    return p;
}

// Slots per lane and warps per SM.  With the hi/lo displacement eight slots a
// lane (8 warps, 240 registers) amortise the shuffles best once there are
// enough steps for every warp; below, the smaller blocks of four slots (12
// warps) start and finish faster (F64ACC evaluation, eight / four: 56.4 / 52.3
// us at 8192, 67.5 / 64.6 at 10000, 89.3 / 90.9 at 12288, 109.2 / 116.0 at
// 14336, 485 / 515 at 32768).  Single-float displacements need
// fewer registers, and 16 warps of four slots hide more latency at every
// size: 111.0 / 102.8 us at 16384.
constexpr int64_t kWideBlockMinN = 12288;

template <bool POT, bool F64>
int launch_pair_shape(Params &p, bool split, cudaStream_t st) {
    if (!split) return launch_pairs<ForcePh<false, 4, 16, false, POT>, F64>(p, st);
    return p.N >= kWideBlockMinN ? launch_pairs<ForcePh<false, 8, 8, true, POT>, F64>(p, st)
                                 : launch_pairs<ForcePh<false, 4, 12, true, POT>, F64>(p, st);
}

int launch_pair_kernel(const ForceJob &j, Params &p, bool pot) {
    const bool f64 = j.precision == NB_PREC_F64ACC;
    kernel_timer_begin(j.stream);
    const int rc = pot ? (f64 ? launch_pair_shape<true, true>(p, j.split, j.stream)
                              : launch_pair_shape<true, false>(p, j.split, j.stream))
                       : (f64 ? launch_pair_shape<false, true>(p, j.split, j.stream)
                              : launch_pair_shape<false, false>(p, j.split, j.stream));
    kernel_timer_end(j.stream);
    return rc;
}

int launch_wsym_pack(const ForceJob &j, double *vel, double kick, double drift) {
    const int nc = j.pot ? 4 : 3;
    return launch_pdl(wsym_pack_kernel, pack_blocks(j.L.Np, j.N, nc), 128, 0, j.stream,
                      const_cast<double *>(j.pos), vel, j.acc, j.mass, j.N, j.L.Np, kick, drift,
                      reinterpret_cast<float *>(j.ws + j.L.packA), maxima(j),
                      reinterpret_cast<unsigned long long *>(j.ws + j.L.wsym_fx), nc);
}

int launch_wsym_fold(const ForceJob &j, const Params &p, double *pot, bool next, double *vel,
                     double kick, double next_kick, double drift) {
    const unsigned blocks = (unsigned)cdiv(j.N, 128);
    auto k = next ? wsym_fold_kernel<true> : wsym_fold_kernel<false>;
    return launch_pdl(k, blocks, 128, 0, j.stream, p, j.G, j.acc, pot,
                      const_cast<double *>(j.pos), vel, kick, next_kick, drift,
                      reinterpret_cast<float *>(j.ws + j.L.packA), maxima(j));
}

}  // namespace

int launch_force_wsym(const ForceJob &j) {
    Params p = params_of(j);
    int rc = launch_wsym_pack(j, nullptr, 0.0, 0.0);
    if (rc) return rc;
    if ((rc = launch_pair_kernel(j, p, j.pot != nullptr))) return rc;
    return launch_wsym_fold(j, p, j.pot, false, j.vel, j.kick, 0.0, 0.0);
}

int launch_step_wsym(const ForceJob &j, double *vel, double dt, int64_t nsteps, bool acc_valid) {
    Params p = params_of(j);
    const double half = 0.5 * dt;
    int rc = launch_wsym_pack(j, acc_valid ? vel : nullptr, half, dt);
    if (rc) return rc;
    // evaluation e = 0 is the priming one when a(x) is not known yet
    for (int64_t e = acc_valid ? 1 : 0; e <= nsteps; ++e) {
        const bool next = e < nsteps;
        double *pot = next ? nullptr : j.pot;
        if ((rc = launch_pair_kernel(j, p, pot != nullptr))) return rc;
        if ((rc = launch_wsym_fold(j, p, pot, next, nsteps ? vel : nullptr, e ? half : 0.0, half,
                                   dt)))
            return rc;
    }
    return NB_OK;
}

}  // namespace nb
