// k_marg.cu -- the exact x-marginal p(x) = WHT(WHT(q)^2) s^2 / d, q = |psi|^2,
// with its transforms in 64-bit integers.
//
// FP64 additions issue at 2 per clock and SM on this part, 64-bit integer ones
// (two 32-bit instructions) at about 32. A pass therefore reads doubles, turns
// the numbers of its tile into integers times one power of two, transforms
// those exactly, and writes doubles again. Per pass a number is rounded twice,
// once to the tile's quantum and once back to 53 bits, instead of once per
// transform stage. The quantum is 2^-62 times (less than twice) the largest sum
// of magnitudes over one transform of the tile, so no sum can overflow; strided
// passes of K < 4 bits (N = 13 to 15) take the magnitudes of 2^(4-K) columns
// together, a quantum up to eight times that and still 2^-58 of the column's sum.
// Over at most 11 bits it rounds random data no worse than 11 FP64 stages do
// (measured against extended precision, N = 13 to 22: not above the FP64 passes'
// error).
//
// The transforms are packed: element g < 2^n (n = N - 1) holds the pair
// (value(g), value(g + d/2)), two real transforms side by side, and the top bit
// is the sum and difference of the pair. A marginal is
//   strided passes (psi -> q on the first), from the top bits down to bit 11;
//   the row pass: bits 10..0, the pair's sum and difference, the square, and
//     bits 0..10 again;
//   the strided passes once more, the last one writing p.
// Tiles are 2^12 pairs (64 KB), 256 threads x 16 pairs: two per SM. The row pass
// in the middle saves one trip through memory.
//
// N = 27 (2^27 numbers, 1 GB), without the norm that both need (0.23 ms): 16.2 ms
// with FP64 passes (FP64 pipe 76-83% busy), 2.9 ms with these; whole calls 17.2 and
// 3.2 ms.
#include "k_misc.cuh"
#include "k_fp64.cuh"

namespace sre {

namespace {

constexpr int MB = 12;                     // tile bits
constexpr int MR = MARG_ROW_BITS;          // row bits
constexpr int MT = 256;                    // threads
typedef long long i64;
struct __align__(16) Pair { i64 x, y; };

__host__ __device__ constexpr uint32_t mphys(uint32_t e) { return e + (e >> 4); }
constexpr size_t MARG_SMEM = sizeof(Pair) * (size_t)mphys(1u << MB) + sizeof(float) * (4 * MT + 32);

// element of (thread t, slot k) when the slot bits start at a
__device__ __forceinline__ uint32_t melem(uint32_t t, uint32_t k, int a) {
    return (t & ((1u << a) - 1u)) | (k << a) | ((t >> a) << (a + 4));
}

// |v| rounded up to 20 bits, as a float (0 below 2^-126; the callers' numbers
// stay below 2^127)
__device__ __forceinline__ float mag(double v) {
    const unsigned hi = (unsigned)__double2hiint(v) & 0x7fffffffu;
    return hi < (897u << 20) ? 0.f : __uint_as_float(((hi - (896u << 20)) << 3) | 7u);
}

__device__ __forceinline__ unsigned long long shr64(unsigned long long v, unsigned n) {
    unsigned long long r;
    asm("shr.b64 %0, %1, %2;" : "=l"(r) : "l"(v), "r"(n));    // n > 63 gives 0
    return r;
}

// round(v 2^E), |v| 2^E < 2^62
__device__ __forceinline__ i64 fix(double v, int E) {
    const unsigned hi = (unsigned)__double2hiint(v);
    const int ex = (int)((hi >> 20) & 0x7ffu);
    unsigned long long m = ((unsigned long long)((hi & 0xfffffu) | 0x100000u) << 32) | (unsigned)__double2loint(v);
    if (ex == 0) m = 0;
    const unsigned long long u = (shr64(m << 10, (unsigned)(1084 - ex - E)) + 1ULL) >> 1;
    const i64 s = (i64)((int)hi >> 31);
    return ((i64)u ^ s) - s;
}

// round(f^2 2^E), f^2 2^E < 2^62
__device__ __forceinline__ i64 fix_sq(float f, int E) {
    const unsigned b = __float_as_uint(f);
    const int ex = (int)((b >> 23) & 0xffu);
    const unsigned m = ex ? (b & 0x7fffffu) | 0x800000u : 0u;
    const unsigned long long w = ((unsigned long long)m * m) << 16;
    return (i64)((shr64(w, (unsigned)(315 - 2 * ex - E)) + 1ULL) >> 1);     // m^2 2^(2 ex - 300)
}

// X 2^-E rounded to 53 bits, by the conversion instruction (FP64 pipe) ...
__device__ __forceinline__ double unfix(i64 X, int E) {
    const double v = __ll2double_rn(X);
    return X ? __hiloint2double(__double2hiint(v) - (E << 20), __double2loint(v)) : 0.0;
}
// ... and in integer operations (halves away from zero). The row pass and the
// last pass use one for each number of a pair, so that neither pipe waits for
// the other: 2.87 ms in all at N = 27, against 3.21 with the conversion alone
// and 2.93 without it.
__device__ __forceinline__ double unfix_alu(i64 X, int E) {
    const unsigned long long u = X < 0 ? 0ULL - (unsigned long long)X : (unsigned long long)X;
    const int z = __clzll((i64)u);
    const unsigned long long w = u << (z & 63);
    const unsigned long long m = (w >> 11) + ((w >> 10) & 1ULL);          // 2^52 .. 2^53
    const int hi = (int)(m >> 32) + ((1085 - z - E) << 20);               // the leading bit adds one to the exponent
    return X ? __hiloint2double(hi | ((int)(X >> 32) & (int)0x80000000), (int)m) : 0.0;
}

// quantum exponent for sums of magnitudes up to S: S 2^E < 2^62
__device__ __forceinline__ int exponent(float S) {
    const unsigned b = __float_as_uint(S * 1.0001f);     // the sums of S round by less
    return b == 0u ? 0 : 61 - ((int)(b >> 23) - 127);
}

// maximum over the CTA of non-negative floats; scratch: 8 words. Two barriers.
__device__ __forceinline__ float block_max(float v, unsigned *scratch) {
    const unsigned w = __reduce_max_sync(0xffffffffu, __float_as_uint(v));
    __syncthreads();
    if ((threadIdx.x & 31) == 0) scratch[threadIdx.x >> 5] = w;
    __syncthreads();
    unsigned m = 0;
#pragma unroll
    for (int i = 0; i < MT / 32; ++i) m = max(m, scratch[i]);
    return __uint_as_float(m);
}

// largest sum over the threads that agree in the low c bits of t (c <= 8), of
// the two values of each thread; sh: 2 MT floats + 8 words
__device__ __forceinline__ float max_column_sum(float a, float b, int c, float *sh) {
    for (int o = 1 << c; o < 32; o <<= 1) {
        a += __shfl_xor_sync(0xffffffffu, a, o);
        b += __shfl_xor_sync(0xffffffffu, b, o);
    }
    const int t = threadIdx.x;
    sh[t] = a;
    sh[MT + t] = b;
    __syncthreads();
    const int step = c < 5 ? 32 : 1 << c, first = t & (step - 1);
    float sa = 0.f, sb = 0.f;
    for (int i = first; i < MT; i += step) {
        sa += sh[i];
        sb += sh[MT + i];
    }
    return block_max(fmaxf(sa, sb), reinterpret_cast<unsigned *>(sh + 2 * MT));
}

template <int S0, int S1>
__device__ __forceinline__ void stages(Pair (&v)[16]) {
#pragma unroll
    for (int s = S0; s < S1; ++s)
#pragma unroll
        for (int k = 0; k < 16; ++k)
            if (!(k & (1 << s))) {
                const Pair a = v[k], b = v[k | (1 << s)];
                v[k].x = a.x + b.x;
                v[k].y = a.y + b.y;
                v[k | (1 << s)].x = a.x - b.x;
                v[k | (1 << s)].y = a.y - b.y;
            }
}

template <int A, int B>
__device__ __forceinline__ void exchange(Pair (&v)[16], Pair *sm, uint32_t t) {
    Pair *p = sm + mphys(melem(t, 0, A));
#pragma unroll
    for (int k = 0; k < 16; ++k) p[mphys((uint32_t)k << A)] = v[k];
    __syncthreads();
    const Pair *q = sm + mphys(melem(t, 0, B));
#pragma unroll
    for (int k = 0; k < 16; ++k) v[k] = q[mphys((uint32_t)k << B)];
}

enum { MS_PSI = 0, MS_BUF = 1 };
enum { MD_BUF = 0, MD_P = 1 };

// Power of two h with sum |psi|^2 4^h in (1/4, 1]: psi 2^h is summed without
// overflow or harmful underflow in the FP32 magnitudes.
__device__ __forceinline__ int psi_shift(double s) {
    const int ex = (int)(((unsigned)__double2hiint(s) >> 20) & 0x7ffu) - 1023;     // s = 1 / sum |psi|^2
    const int h = ex >> 1;
    return h < -126 ? -126 : h > 126 ? 126 : h;
}

// K bits from lo on: tiles of 2^K rows x 2^(12-K) columns
template <int K, int SRC, int DST>
__global__ void __launch_bounds__(MT, 2) marg_strided(const float2 *psi, const double2 *src, double2 *dst, double *p, int n,
                                                      int lo, const double *scal) {
    extern __shared__ __align__(16) unsigned char smraw[];
    Pair *sm = reinterpret_cast<Pair *>(smraw);
    float *sh = reinterpret_cast<float *>(smraw + sizeof(Pair) * (size_t)mphys(1u << MB));
    constexpr int C = MB - K;
    const uint32_t t = threadIdx.x;
    const uint32_t tile = blockIdx.x, cbits = (uint32_t)(lo - C);
    const uint32_t gb = ((tile >> cbits) << (lo + K)) | ((tile & ((1u << cbits) - 1u)) << C);
    auto gidx = [&](uint32_t e) { return gb | ((e >> C) << lo) | (e & ((1u << C) - 1u)); };
    const uint32_t half = 1u << n;
    constexpr int A0 = 8;
    Pair v[16];
    int E;
    if constexpr (SRC == MS_PSI) {
        const float f = __uint_as_float((unsigned)(psi_shift(scal[SCAL_S]) + 127) << 23);
        float2 u[16], w[16];
        float a = 0.f, b = 0.f;
#pragma unroll
        for (int k = 0; k < 16; ++k) {
            const uint32_t g = gidx(melem(t, k, A0));
            u[k] = __ldg(psi + g);
            w[k] = __ldg(psi + (g | half));
        }
#pragma unroll
        for (int k = 0; k < 16; ++k) {
            u[k].x *= f; u[k].y *= f; w[k].x *= f; w[k].y *= f;
            a += fmaf(u[k].x, u[k].x, u[k].y * u[k].y);
            b += fmaf(w[k].x, w[k].x, w[k].y * w[k].y);
        }
        E = exponent(max_column_sum(a, b, C < 8 ? C : 8, sh));
#pragma unroll
        for (int k = 0; k < 16; ++k) {
            v[k].x = fix_sq(u[k].x, E) + fix_sq(u[k].y, E);
            v[k].y = fix_sq(w[k].x, E) + fix_sq(w[k].y, E);
        }
    } else {
        double2 d[16];
        float a = 0.f, b = 0.f;
#pragma unroll
        for (int k = 0; k < 16; ++k) d[k] = src[gidx(melem(t, k, A0))];
#pragma unroll
        for (int k = 0; k < 16; ++k) {
            a += mag(d[k].x);
            b += mag(d[k].y);
        }
        E = exponent(max_column_sum(a, b, C < 8 ? C : 8, sh));
#pragma unroll
        for (int k = 0; k < 16; ++k) {
            v[k].x = fix(d[k].x, E);
            v[k].y = fix(d[k].y, E);
        }
    }
    constexpr int AL = K <= 4 ? 8 : K <= 8 ? 4 : 3;
    stages<(K < 4 ? 4 - K : 0), 4>(v);
    if constexpr (K > 4) {
        exchange<8, 4>(v, sm, t);
        stages<(K < 8 ? 8 - K : 0), 4>(v);
    }
    if constexpr (K > 8) {
        static_assert(K == 9, "strided passes of at most nine bits");
        exchange<4, 3>(v, sm, t);
        stages<0, 1>(v);
    }
    if constexpr (DST == MD_BUF) {
#pragma unroll
        for (int k = 0; k < 16; ++k) dst[gidx(melem(t, k, AL))] = make_double2(unfix(v[k].x, E), unfix(v[k].y, E));
    } else {
        // p = s^2 / d of the sums, with the 4^h that psi carried taken out; a
        // norm that is not finite leaves no number here
        const double s = scal[SCAL_S];
        double f = __hiloint2double((1023 - 2 * psi_shift(s)) << 20, 0) * s;
        f = f * f * (0.5 / (double)half);
        if (!(scal[SCAL_NORM2] <= 1.7976931348623157e308)) f = __longlong_as_double(0x7ff8000000000000LL);
#pragma unroll
        for (int k = 0; k < 16; ++k) {
            const uint32_t g = gidx(melem(t, k, AL));
            p[g] = unfix(v[k].x + v[k].y, E) * f;
            p[g | half] = unfix_alu(v[k].x - v[k].y, E) * f;
        }
    }
}

// bits 10..0 of the first transform, its top bit, the square, and bits 0..10
// of the second; two rows of 2^11 per tile (tile bit 11), in place
__global__ void __launch_bounds__(MT, 2) marg_row(double2 *buf) {
    extern __shared__ __align__(16) unsigned char smraw[];
    Pair *sm = reinterpret_cast<Pair *>(smraw);
    float *sh = reinterpret_cast<float *>(smraw + sizeof(Pair) * (size_t)mphys(1u << MB));
    const uint32_t t = threadIdx.x;
    double2 *row = buf + ((size_t)blockIdx.x << MB);
    Pair v[16];
    int E;
    {
        double2 d[16];
        float a[2] = {0.f, 0.f}, b[2] = {0.f, 0.f};
#pragma unroll
        for (int k = 0; k < 16; ++k) d[k] = row[melem(t, k, 8)];
#pragma unroll
        for (int k = 0; k < 16; ++k) {
            a[k >> 3] += mag(d[k].x);
            b[k >> 3] += mag(d[k].y);
        }
        // the rows are slots 0-7 and 8-15 of every thread
#pragma unroll
        for (int o = 16; o > 0; o >>= 1)
#pragma unroll
            for (int r = 0; r < 2; ++r) {
                a[r] += __shfl_xor_sync(0xffffffffu, a[r], o);
                b[r] += __shfl_xor_sync(0xffffffffu, b[r], o);
            }
        if ((t & 31) == 0) {
            float *o = sh + 4 * (t >> 5);
            o[0] = a[0]; o[1] = a[1]; o[2] = b[0]; o[3] = b[1];
        }
        __syncthreads();
        float S = 0.f;
#pragma unroll
        for (int r = 0; r < 4; ++r) {
            float q = 0.f;
#pragma unroll
            for (int w = 0; w < MT / 32; ++w) q += sh[4 * w + r];
            S = fmaxf(S, q);
        }
        E = exponent(S);
#pragma unroll
        for (int k = 0; k < 16; ++k) {
            v[k].x = fix(d[k].x, E);
            v[k].y = fix(d[k].y, E);
        }
    }
    stages<0, 3>(v);
    exchange<8, 4>(v, sm, t);
    stages<0, 4>(v);
    exchange<4, 0>(v, sm, t);
    stages<0, 4>(v);
    {
        double2 d[16];
        float a = 0.f, b = 0.f;
#pragma unroll
        for (int k = 0; k < 16; ++k) {
            const double x = unfix(v[k].x + v[k].y, E), y = unfix_alu(v[k].x - v[k].y, E);
            d[k] = make_double2(x * x, y * y);
            a += mag(d[k].x);
            b += mag(d[k].y);
        }
        // slots are bits 0-3 now: a row is four warps
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            a += __shfl_xor_sync(0xffffffffu, a, o);
            b += __shfl_xor_sync(0xffffffffu, b, o);
        }
        float *so = sh + 64;                       // apart from the first sums, which others may still read
        if ((t & 31) == 0) {
            so[t >> 5] = a;
            so[8 + (t >> 5)] = b;
        }
        __syncthreads();
        float S = 0.f;
#pragma unroll
        for (int r = 0; r < 4; ++r) {
            float q = 0.f;
#pragma unroll
            for (int w = 0; w < 4; ++w) q += so[4 * r + w];
            S = fmaxf(S, q);
        }
        E = exponent(S);
#pragma unroll
        for (int k = 0; k < 16; ++k) {
            v[k].x = fix(d[k].x, E);
            v[k].y = fix(d[k].y, E);
        }
    }
    stages<0, 4>(v);
    exchange<0, 4>(v, sm, t);
    stages<0, 4>(v);
    exchange<4, 8>(v, sm, t);
    stages<0, 3>(v);
#pragma unroll
    for (int k = 0; k < 16; ++k) row[melem(t, k, 8)] = make_double2(unfix(v[k].x, E), unfix_alu(v[k].y, E));
}

template <int K, int SRC, int DST>
cudaError_t strided(const float2 *psi, double2 *buf, double *p, int n, int lo, const double *scal, cudaStream_t st) {
    static SmemOptIn optin;
    const cudaError_t e = optin.allow((const void *)marg_strided<K, SRC, DST>, MARG_SMEM);
    if (e != cudaSuccess) return e;
    marg_strided<K, SRC, DST><<<1u << (n - MB), MT, MARG_SMEM, st>>>(psi, buf, buf, p, n, lo, scal);
    return cudaGetLastError();
}

template <int SRC, int DST>
cudaError_t strided_k(int K, const float2 *psi, double2 *buf, double *p, int n, int lo, const double *scal,
                      cudaStream_t st) {
    switch (K) {
#define C(k) case k: return strided<k, SRC, DST>(psi, buf, p, n, lo, scal, st);
    C(1) C(2) C(3) C(4) C(5) C(6) C(7) C(8) C(9)
#undef C
    default: return cudaErrorInvalidValue;
    }
}

} // namespace

cudaError_t launch_marginal(const float2 *psi, int N, const double *scal, double *p, double *work, int *launches,
                            cudaStream_t st) {
    const int n = N - 1, rest = n - MR;
    if (rest < 1 || n > 29) return cudaErrorInvalidValue;
    const int ns = (rest + MARG_STRIDED_MAX - 1) / MARG_STRIDED_MAX;
    double2 *buf = reinterpret_cast<double2 *>(work);
    int K[2], lo[2], top = n;
    for (int i = 0; i < ns; ++i) {
        K[i] = rest / ns + (i >= ns - rest % ns ? 1 : 0);
        top -= K[i];
        lo[i] = top;
    }
    cudaError_t e;
    for (int i = 0; i < ns; ++i) {
        e = i == 0 ? strided_k<MS_PSI, MD_BUF>(K[i], psi, buf, p, n, lo[i], scal, st)
                   : strided_k<MS_BUF, MD_BUF>(K[i], psi, buf, p, n, lo[i], scal, st);
        if (e != cudaSuccess) return e;
    }
    static SmemOptIn optin;
    e = optin.allow((const void *)marg_row, MARG_SMEM);
    if (e != cudaSuccess) return e;
    marg_row<<<1u << (n - MB), MT, MARG_SMEM, st>>>(buf);
    e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    for (int i = ns - 1; i >= 0; --i) {
        e = i == 0 ? strided_k<MS_BUF, MD_P>(K[i], psi, buf, p, n, lo[i], scal, st)
                   : strided_k<MS_BUF, MD_BUF>(K[i], psi, buf, p, n, lo[i], scal, st);
        if (e != cudaSuccess) return e;
    }
    *launches = 2 * ns + 1;
    return cudaSuccess;
}

} // namespace sre
