// Space-filling-curve order of particles: the cell of a coordinate, its
// Hilbert index, and a CTA-wide bitonic sort of 64-bit keys in shared
// memory.  A Hilbert curve has no jumps between neighbouring indices, so a
// run of consecutive particles is spatially more compact than along a Morton
// (Z-order) curve: fewer overlapping boxes, fewer near (hi/lo) j-sets.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

namespace nb {
namespace dev {

// Spreads the low 10 bits of v so that bit k lands at bit 3k.
__device__ __forceinline__ uint32_t spread3(uint32_t v) {
    uint32_t r = 0;
#pragma unroll
    for (int k = 0; k < 10; ++k) r |= ((v >> k) & 1u) << (3 * k);
    return r;
}

// Index of the cell (x, y, z) (10 bits each) along a 3D Hilbert curve,
// 30 bits: J. Skilling's transposition method (Programming the Hilbert
// curve, AIP Conf. Proc. 707, 2004) -- undo the excess work level by level
// (invert or exchange the low bits), Gray-encode across the axes, then
// interleave the transposed bits with the first axis most significant.
__device__ __forceinline__ uint32_t hilbert30(uint32_t x, uint32_t y, uint32_t z) {
    uint32_t X[3] = {x, y, z};
    for (uint32_t Q = 1u << 9; Q > 1; Q >>= 1) {
        const uint32_t P = Q - 1;
#pragma unroll
        for (int i = 0; i < 3; ++i) {
            if (X[i] & Q) {
                X[0] ^= P;
            } else {
                const uint32_t t = (X[0] ^ X[i]) & P;
                X[0] ^= t;
                X[i] ^= t;
            }
        }
    }
    X[1] ^= X[0];
    X[2] ^= X[1];
    uint32_t t = 0;
    for (uint32_t Q = 1u << 9; Q > 1; Q >>= 1)
        if (X[2] & Q) t ^= Q - 1;
#pragma unroll
    for (int i = 0; i < 3; ++i) X[i] ^= t;
    return (spread3(X[0]) << 2) | (spread3(X[1]) << 1) | spread3(X[2]);
}

// The cell of one coordinate: (x - lo) * scale truncated and clamped to [0,
// 1023] (as an integer: the conversion saturates, and FP64 compares are slow on
// this part).
__device__ __forceinline__ uint32_t cell10(double x, double lo, double scale) {
    const int q = __double2int_rz((x - lo) * scale);
    return (uint32_t)min(max(q, 0), 1023);
}

// Order-preserving image of a double as a signed integer, and back.
__device__ __forceinline__ long long ordered_bits(double x) {
    const long long b = __double_as_longlong(x);
    return b >= 0 ? b : (b ^ 0x7fffffffffffffffLL);
}
__device__ __forceinline__ double from_ordered(long long b) {
    return __longlong_as_double(b >= 0 ? b : (b ^ 0x7fffffffffffffffLL));
}

// Ascending bitonic sort of P (a power of two) 64-bit keys in shared memory
// by the whole CTA (every thread calls it; it ends with a barrier).
__device__ __forceinline__ void block_bitonic_sort(unsigned long long *keys, int P) {
    for (int k = 2; k <= P; k <<= 1)
        for (int j = k >> 1; j > 0; j >>= 1) {
            for (int e = threadIdx.x; e < P; e += blockDim.x) {
                const int x = e ^ j;
                if (x > e) {
                    const bool asc = (e & k) == 0;
                    const unsigned long long a = keys[e], b = keys[x];
                    if ((a > b) == asc) {
                        keys[e] = b;
                        keys[x] = a;
                    }
                }
            }
            __syncthreads();
        }
}

// Ascending bitonic sort of T E 64-bit keys by a CTA of T threads (every thread
// calls it).  Thread t holds elements t E .. t E + E - 1 in registers: strides
// below E are exchanges within the thread, strides below 32 E shuffles within
// the warp, and only the longer ones (10 of the 91 stages of 8192 keys) go
// through shared memory, where block_bitonic_sort takes every stage there with
// a barrier each.  keys: in linear order on entry and, after the barrier at
// the end, on exit.
// Only the stages k_lo .. k_hi, with directions from the elements' global index
// base + ..., when the keys are a chunk of a longer sequence (strides of a chunk
// or more are done elsewhere).
template <int T, int E>
__device__ __forceinline__ void block_sort_regs(unsigned long long *keys, int64_t k_lo = 2,
                                                int64_t k_hi = T * E, int64_t base = 0) {
    const int t = threadIdx.x;
    unsigned long long v[E];
#pragma unroll
    for (int e = 0; e < E; ++e) v[e] = keys[t * E + e];
    __syncthreads();
    // keeps the smaller of own and other on the lower side of an ascending run
    auto keep = [](unsigned long long own, unsigned long long other, bool small) {
        return (own < other) == small ? own : other;
    };
    for (int64_t k = k_lo; k <= k_hi; k <<= 1) {
        for (int j = k >= T * E ? T * E / 2 : (int)(k >> 1); j >= E; j >>= 1) {
            const int m = j / E;
            const bool lower = !(t & m);
            if (m >= 32) {  // the shared copy is [E][T]: no bank conflicts
#pragma unroll
                for (int e = 0; e < E; ++e) keys[e * T + t] = v[e];
                __syncthreads();
#pragma unroll
                for (int e = 0; e < E; ++e) {
                    const bool asc = ((base + t * E + e) & k) == 0;
                    v[e] = keep(v[e], keys[e * T + (t ^ m)], lower == asc);
                }
                __syncthreads();
            } else {
#pragma unroll
                for (int e = 0; e < E; ++e) {
                    const bool asc = ((base + t * E + e) & k) == 0;
                    v[e] = keep(v[e], __shfl_xor_sync(0xffffffffu, v[e], m), lower == asc);
                }
            }
        }
#pragma unroll
        for (int j = E / 2; j > 0; j >>= 1)
            if (j < k) {
#pragma unroll
                for (int e = 0; e < E; ++e)
                    if (!(e & j)) {
                        const bool asc = ((base + t * E + e) & k) == 0;
                        const unsigned long long a = v[e], b = v[e + j];
                        const bool swap = (a > b) == asc;
                        v[e] = swap ? b : a;
                        v[e + j] = swap ? a : b;
                    }
            }
    }
#pragma unroll
    for (int e = 0; e < E; ++e) keys[t * E + e] = v[e];
    __syncthreads();
}

}  // namespace dev
}  // namespace nb
