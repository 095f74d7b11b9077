// k_fp64.cuh -- FP64 helpers: exact widening of FP32 data, compensated sums.
#pragma once

#include <cuda_runtime.h>

namespace sre {

// binary32 -> binary64 by re-packing the fields (exact: every float is a
// double). The conversion instruction runs on the FP64 pipe, which issues
// one warp instruction per 16 cycles on this part; normal numbers and zeros
// go through integer operations instead, and only subnormals, inf and NaN
// take the instruction.
__device__ __forceinline__ double f2d(float f) {
    const unsigned u = __float_as_uint(f);
    const unsigned e = (u >> 23) & 0xFFu, m = u & 0x7FFFFFu, sg = u & 0x80000000u;
    if (e == 0u && m == 0u) return __hiloint2double((int)sg, 0);
    if (e - 1u >= 254u) return (double)f;
    return __hiloint2double((int)(sg | ((e + 896u) << 20) | (m >> 3)), (int)(m << 29));
}

// Sum of |u|^2 over G amplitudes, to the precision of FP64 additions in integer
// operations (FP64 issues 2 lanes per clock and SM on this part): the squares
// of the 24-bit significands are aligned to the group's largest exponent in
// units of 2^-11 of their last bit and added as 64-bit integers; a term loses
// less than 2^-57 of the group's sum. Groups that hold inf or NaN, or nothing
// above 2^-63, take the FP64 operations.
template <int G>
__device__ __forceinline__ double sum_squares(const float2 (&u)[G]) {
    static_assert(G <= 8, "16 squares below 2^59 each");
    unsigned top = 0;
#pragma unroll
    for (int k = 0; k < G; ++k) {
        top = max(top, __float_as_uint(u[k].x) & 0x7fffffffu);
        top = max(top, __float_as_uint(u[k].y) & 0x7fffffffu);
    }
    const int E = (int)(top >> 23);
    if (E == 255 || E < 64) {
        double acc = 0.0;
#pragma unroll 1
        for (int k = 0; k < G; ++k) {
            const double x = f2d(u[k].x), y = f2d(u[k].y);
            acc = fma(x, x, acc);
            acc = fma(y, y, acc);
        }
        return acc;
    }
    unsigned long long sum = 0;
#pragma unroll
    for (int k = 0; k < 2 * G; ++k) {
        const unsigned b = __float_as_uint(k & 1 ? u[k / 2].y : u[k / 2].x);
        const unsigned m = (b & 0x7fffffu) | 0x800000u;
        const unsigned sh = (unsigned)(2 * (E - (int)((b >> 23) & 0xffu)));   // zeros and subnormals: >= 128
        unsigned long long q;
        asm("shr.b64 %0, %1, %2;" : "=l"(q) : "l"(((unsigned long long)m * m) << 11), "r"(sh));   // 0 from 64 on
        sum += q;
    }
    return (double)sum * __hiloint2double((1023 + 2 * (E - 150) - 11) << 20, 0);
}

// Neumaier's compensated summation (Neumaier 1974, the Kahan-Babuska form):
// s is the running sum and c gathers the rounding error of every addition,
// so s + c carries a sum of many terms to about one rounding of the result.
struct NeuSum {
    double s = 0.0, c = 0.0;
    __device__ __forceinline__ void add(double x) {
        const double t = s + x;
        c += (fabs(s) >= fabs(x)) ? ((s - t) + x) : ((x - t) + s);
        s = t;
    }
    __device__ __forceinline__ double value() const { return s + c; }
};

// Sums over a warp of V values per lane (V a power of two up to 32) by recursive
// halving: each step hands half of the values to the partner lane, so the warp
// issues V - 1 + (5 - log2 V) additions instead of 5 V. Returns the total of
// value id (set per lane; lanes that share an id hold the same total).
template <int V>
__device__ __forceinline__ double warp_sums(double (&v)[V], int &id) {
    static_assert(V >= 1 && V <= 32 && (V & (V - 1)) == 0, "a power of two");
    const int lane = threadIdx.x & 31;
    id = 0;
    int o = 16;
#pragma unroll
    for (int w = V / 2; w >= 1; w /= 2) {
        const bool up = lane & o;
#pragma unroll
        for (int i = 0; i < w; ++i) {
            const double send = up ? v[i] : v[i + w], keep = up ? v[i + w] : v[i];
            v[i] = keep + __shfl_xor_sync(0xffffffffu, send, o);
        }
        id |= up ? w : 0;
        o >>= 1;
    }
    for (; o > 0; o >>= 1) v[0] += __shfl_xor_sync(0xffffffffu, v[0], o);
    return v[0];
}

}  // namespace sre
