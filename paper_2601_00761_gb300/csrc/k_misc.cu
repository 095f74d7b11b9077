// k_misc.cu -- normalisation, reductions, the FP64 CDF scan, Philox draws,
// the two-level z sampler and the MC statistics.
#include "k_misc.cuh"
#include "k_pass_dispatch.cuh"
#include "k_fp64.cuh"

namespace sre {

// ------------------------------------------------------------------ Philox
// Philox4x64-10 (Salmon, Moraes, Dror, Shaw, SC'11): ten rounds of
// (hi, lo) = M * c products with a Weyl key schedule.
__device__ __forceinline__ void philox4x64_10(unsigned long long c[4], unsigned long long k0,
                                              unsigned long long k1) {
    const unsigned long long M0 = 0xD2E7470EE14C6C93ULL, M1 = 0xCA5A826395121157ULL;
    const unsigned long long W0 = 0x9E3779B97F4A7C15ULL, W1 = 0xBB67AE8584CAA73BULL;
#pragma unroll
    for (int r = 0; r < 10; ++r) {
        if (r) { k0 += W0; k1 += W1; }
        const unsigned long long hi0 = __umul64hi(M0, c[0]), lo0 = M0 * c[0];
        const unsigned long long hi1 = __umul64hi(M1, c[2]), lo1 = M1 * c[2];
        const unsigned long long n0 = hi1 ^ c[1] ^ k0, n2 = hi0 ^ c[3] ^ k1;
        c[0] = n0; c[1] = lo1; c[2] = n2; c[3] = lo0;
    }
}

// Uniform of stream (seed), counter (ctr0 + i, lane, 0, 0): word 0, 53 bits.
__device__ __forceinline__ double mc_uniform(unsigned long long seed, unsigned long long ctr0,
                                             unsigned long long i, unsigned long long lane) {
    unsigned long long c[4] = {ctr0 + i, lane, 0ULL, 0ULL};
    philox4x64_10(c, seed, 0ULL);
    return (double)(c[0] >> 11) * 0x1.0p-53;
}

__global__ void philox_test_kernel(const unsigned long long *ctr_key, unsigned long long *out, int n) {
    int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    unsigned long long c[4] = {ctr_key[6 * i], ctr_key[6 * i + 1], ctr_key[6 * i + 2], ctr_key[6 * i + 3]};
    philox4x64_10(c, ctr_key[6 * i + 4], ctr_key[6 * i + 5]);
    for (int w = 0; w < 4; ++w) out[4 * i + w] = c[w];
}

// ------------------------------------------------------------ reductions
template <int NT>
__device__ __forceinline__ double block_sum(double v, double *red) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    __syncthreads();
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = v;
    __syncthreads();
    double s = 0.0;
    if (threadIdx.x == 0)
        for (int w = 0; w < NT / 32; ++w) s += red[w];
    return s;
}

// A thread's part of sum |psi|^2: amplitudes first, first + stride, ... below d
// in groups of eight, all of a group's loads in flight.
__device__ __forceinline__ double norm2_part(const float2 *psi, unsigned long long d, unsigned long long first,
                                             unsigned long long stride) {
    constexpr int G = 8;
    double acc = 0.0;
    for (unsigned long long b = first; b < d; b += G * stride) {
        float2 u[G];
#pragma unroll
        for (int k = 0; k < G; ++k)
            u[k] = b + k * stride < d ? __ldg(psi + b + k * stride) : make_float2(0.f, 0.f);
        acc += sum_squares<G>(u);
    }
    return acc;
}

__device__ __forceinline__ void norm2_write(double n2, double *scal) {
    scal[SCAL_NORM2] = n2;
    scal[SCAL_S] = n2 > 0.0 ? 1.0 / n2 : 0.0;
}

// sum |psi|^2: fixed grid, per-block partials (partial), or one block (scal).
// With FP64 squares the FP64 pipe bound it (N = 27 1002 us, N = 24 133 us); now
// memory does (N = 27 225 us, 4.8 TB/s; N = 24 32 us)
template <bool ONE>
__global__ void __launch_bounds__(256) norm2_partial_kernel(const float2 *psi, unsigned long long d, double *out,
                                                            unsigned long long *zero) {
    __shared__ double red[8];
    const double acc = block_sum<256>(norm2_part(psi, d, (unsigned long long)blockIdx.x * 256 + threadIdx.x,
                                                 (unsigned long long)gridDim.x * 256), red);
    if (zero && blockIdx.x == 0 && threadIdx.x < 2) zero[threadIdx.x] = 0ULL;
    if (threadIdx.x == 0) {
        if constexpr (ONE) norm2_write(acc, out);
        else out[blockIdx.x] = acc;
    }
}

__global__ void __launch_bounds__(256) norm2_final_kernel(const double *partial, int np, double *scal) {
    __shared__ double red[8];
    double acc = 0.0;
    for (int i = threadIdx.x; i < np; i += 256) acc += partial[i];
    acc = block_sum<256>(acc, red);
    if (threadIdx.x == 0) norm2_write(acc, scal);
}

cudaError_t launch_norm2(const float2 *psi, int N, double *scal, double *partial, cudaStream_t st, int *launches,
                         unsigned long long *zero) {
    const unsigned long long d = 1ULL << N;
    // one block takes 4.8 us at N = 10 (32 amplitudes a thread at N = 13), two launches 7.7 us
    if (N <= NORM_ONE_NMAX) {
        norm2_partial_kernel<true><<<1, 256, 0, st>>>(psi, d, scal, zero);
        *launches = 1;
        return cudaGetLastError();
    }
    int nb = NORM_BLOCKS;
    if ((unsigned long long)nb * 2048ULL > d) nb = (int)((d + 2047) / 2048);
    norm2_partial_kernel<false><<<nb, 256, 0, st>>>(psi, d, partial, zero);
    norm2_final_kernel<<<1, 256, 0, st>>>(partial, nb, scal);
    *launches = 2;
    return cudaGetLastError();
}

// tile partials -> family sums; z-range weights scattered to W[fam][range]
__global__ void __launch_bounds__(256) fam_reduce_kernel(const TilePartial *tp, long long n_fam, int tiles,
                                                         const unsigned long long *xs, long long fam_base,
                                                         int N, int M_last, int RL, FamMoments *fm,
                                                         long long fm_base, float *W, long long nr,
                                                         const unsigned long long *perm) {
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const long long f = (long long)blockIdx.x * 8 + warp;
    if (f >= n_fam) return;
    const int n = N - 1;
    unsigned long long x = xs ? xs[fam_base + f] : (unsigned long long)(fam_base + f);
    x &= (1ULL << N) - 1ULL;
    const int j = x ? 63 - __clzll((long long)x) : n;
    // plain FP64: a family's tile partials are FP32 sums (relative error about
    // 1e-7), far above this sum's rounding
    double m[4] = {0.0, 0.0, 0.0, 0.0};
    unsigned c = 0;
    for (int t = lane; t < tiles; t += 32) {
        const TilePartial &p = tp[(size_t)f * tiles + t];
#pragma unroll
        for (int k = 0; k < 4; ++k) m[k] += p.m[k];
        c |= p.cand;
        if (W) {
            const unsigned long long zt = (unsigned long long)t << M_last;
            const unsigned long long rA = insert0(zt, j) >> RL;
            const unsigned long long rB = (j < RL) ? rA + 1 : rA + (1ULL << (j - RL));
            W[(size_t)f * nr + rA] = (float)p.w[0];
            W[(size_t)f * nr + rB] = (float)p.w[1];
        }
    }
    c = __reduce_or_sync(0xffffffffu, c);
    int id;
    const double s = warp_sums<4>(m, id);                // value v in lanes 8 v .. 8 v + 7
    if ((lane & 7) == 0) {
        FamMoments &o = fm[perm ? (long long)perm[fam_base + f] : fm_base + f];
        o.m[id] = s;
        if (lane == 0) o.cand = (unsigned long long)c;
    }
}

// The same sums in the same order for families of many tiles, a warp for each of
// the four values: the chain of a lane's FP64 additions bounds it (2^16 tiles: 2048
// additions). One warp per family for all values takes 20 us for 128 families of
// 2^10 tiles (N = 24) and 920 us for 8 of 2^16 (N = 30); this 7 and 240 us.
__global__ void __launch_bounds__(32) fam_reduce_value_kernel(const TilePartial *tp, int tiles, long long fam_base,
                                                              FamMoments *fm, long long fm_base,
                                                              const unsigned long long *perm) {
    const long long f = blockIdx.y;
    const int k = blockIdx.x, lane = threadIdx.x;
    const TilePartial *row = tp + (size_t)f * (size_t)tiles;
    double v = 0.0;
    unsigned c = 0;
    for (int t0 = 0; t0 < tiles; t0 += 8 * 32) {       // tiles is a power of two, at least 256
        double q[8];
        unsigned b[8];
#pragma unroll
        for (int i = 0; i < 8; ++i) {
            const TilePartial &p = row[t0 + 32 * i + lane];
            q[i] = p.m[k];
            b[i] = k == 0 ? p.cand : 0u;
        }
#pragma unroll
        for (int i = 0; i < 8; ++i) {
            v += q[i];
            c |= b[i];
        }
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    c = __reduce_or_sync(0xffffffffu, c);
    if (lane == 0) {
        FamMoments &o = fm[perm ? (long long)perm[fam_base + f] : fm_base + f];
        o.m[k] = v;
        if (k == 0) o.cand = (unsigned long long)c;
    }
}

cudaError_t launch_fam_reduce(const TilePartial *tp, long long n_fam, int tiles, const unsigned long long *xs,
                              long long fam_base, int N, int M_last, int RL, FamMoments *fm, long long fm_base,
                              float *W, long long nr, cudaStream_t st, const unsigned long long *perm) {
    if (!W && tiles >= 256 && n_fam <= 65535)
        fam_reduce_value_kernel<<<dim3(4, (unsigned)n_fam), 32, 0, st>>>(tp, tiles, fam_base, fm, fm_base, perm);
    else
        fam_reduce_kernel<<<(unsigned)((n_fam + 7) / 8), 256, 0, st>>>(tp, n_fam, tiles, xs, fam_base, N, M_last, RL,
                                                                      fm, fm_base, W, nr, perm);
    return cudaGetLastError();
}

// Totals over the families of each of a run of states: blocks (x) over
// contiguous chunks of a state's families (y), partial sums in the order of the
// families, and the state's last block to finish adds the partials in block
// order, so nothing depends on scheduling. The candidate families go to flags
// (their order is irrelevant: the FP64 counts are integers). FP64 issue bounds
// it; with 1024 blocks whatever the size and one warp-wide sum per value the two
// kernels before took 27 + 20 us for the 1024 families of N = 10 and 38 + 20 us
// for N = 18, one block per state of a batch 175 us: now 11, 15 (N = 16) and 32 us.
__global__ void __launch_bounds__(256) totals_kernel(const TotalsArgs a) {
    __shared__ double red[8][8];
    __shared__ bool last;
    const int st = a.s0 + blockIdx.y, nb = gridDim.x;
    const FamMoments *fm = a.fm + ((((long long)st) << a.N) - a.fm_first);
    const long long n = 1LL << a.N, per = (n + nb - 1) / nb;
    const long long lo = (long long)blockIdx.x * per, hi = lo + per < n ? lo + per : n;
    NeuSum s0, s1, s2, s3, sq;
    for (long long f = lo + threadIdx.x; f < hi; f += 256) {
        const FamMoments m = fm[f];
        s0.add(m.m[0]); s1.add(m.m[1]); s2.add(m.m[2]); s3.add(m.m[3]);
        if (f > 0) sq.add(m.m[1] * m.m[1]);
        if (m.cand && a.flags) a.flags[atomicAdd(a.n_flag, 1ULL)] = ((unsigned long long)st << a.N) | (unsigned long long)f;
    }
    // value v of the block in thread v of warp 0
    auto block_totals = [&](double (&v)[8]) -> double {
        int id;
        const double t = warp_sums<8>(v, id);
        __syncthreads();
        if ((threadIdx.x & 3) == 0) red[threadIdx.x >> 5][id] = t;
        __syncthreads();
        double r = 0.0;
        if (threadIdx.x < 32) {
            const int w = threadIdx.x >> 3, i = threadIdx.x & 7;
            r = red[2 * w][i] + red[2 * w + 1][i];
            r += __shfl_xor_sync(0xffffffffu, r, 8);
            r += __shfl_xor_sync(0xffffffffu, r, 16);
        }
        return r;
    };
    double v[8] = {s0.value(), s1.value(), s2.value(), s3.value(), sq.value(), 0.0, 0.0, 0.0};
    const double t = block_totals(v);
    double *part = a.partial + 5 * ((size_t)blockIdx.y * nb);
    if (nb > 1) {
        if (threadIdx.x < 5) {
            part[5 * (size_t)blockIdx.x + threadIdx.x] = t;
            __threadfence();
        }
        __syncthreads();
        if (threadIdx.x == 0) {
            __threadfence();
            last = atomicAdd(a.done + blockIdx.y, 1u) == (unsigned)nb - 1;
        }
        __syncthreads();
        if (!last) return;
        __threadfence();
        NeuSum q[5];
        for (int i = threadIdx.x; i < nb; i += 256)
#pragma unroll
            for (int k = 0; k < 5; ++k) q[k].add(__ldcg(part + 5 * (size_t)i + k));
#pragma unroll
        for (int k = 0; k < 5; ++k) v[k] = q[k].value();
        v[5] = v[6] = v[7] = 0.0;
        const double u = block_totals(v);
        if (threadIdx.x < 5) a.out[TOT_N * (size_t)st + (threadIdx.x < 4 ? threadIdx.x : 5)] = u;
    } else if (threadIdx.x < 5) {
        a.out[TOT_N * (size_t)st + (threadIdx.x < 4 ? threadIdx.x : 5)] = t;
    }
    if (threadIdx.x == 0) {
        a.out[TOT_N * (size_t)st + 6] = fm[0].m[1];
        if (a.norm2) {
            // every block of the launch's only state has flagged its families
            a.out[TOT_N] = *a.norm2;
            a.out[TOT_N + 1] = a.n_flag ? (double)*reinterpret_cast<volatile unsigned long long *>(a.n_flag) : 0.0;
        }
    }
}

cudaError_t launch_totals(const TotalsArgs &a, int ns, cudaStream_t st) {
    totals_kernel<<<dim3((unsigned)totals_blocks(a.N, ns), (unsigned)ns), 256, 0, st>>>(a);
    return cudaGetLastError();
}

__global__ void sum_u64_kernel(const unsigned long long *v, long long n, unsigned long long *out) {
    __shared__ unsigned long long red[256];
    unsigned long long a = 0;
    for (long long i = threadIdx.x; i < n; i += 256) a += v[i];
    red[threadIdx.x] = a;
    __syncthreads();
    for (int s = 128; s > 0; s >>= 1) {
        if (threadIdx.x < s) red[threadIdx.x] += red[threadIdx.x + s];
        __syncthreads();
    }
    if (threadIdx.x == 0) *out = red[0];
}

cudaError_t launch_sum_u64(const unsigned long long *v, long long n, unsigned long long *out, cudaStream_t st) {
    sum_u64_kernel<<<1, 256, 0, st>>>(v, n, out);
    return cudaGetLastError();
}

// ------------------------------------------------------------- CDF scan
// FP64 sums of p over chunks of SCAN_CHUNK elements, in a fixed association.
__global__ void __launch_bounds__(256) scan_chunk_sums(const double *p, unsigned long long n, double *bsum) {
    __shared__ double red[8];
    const unsigned long long base = (unsigned long long)blockIdx.x * SCAN_CHUNK + threadIdx.x;
    double a = 0.0;
#pragma unroll
    for (int i = 0; i < 16; ++i)
        if (base + 256 * i < n) a += p[base + 256 * i];
    a = block_sum<256>(a, red);
    if (threadIdx.x == 0) bsum[blockIdx.x] = a;
}

// Exclusive prefix of bsum in place within tiles of SCAN_TILE chunks, and the
// total: of the only tile in bsum[nb], else of each in tot.
constexpr long long SCAN_TILE = 8192;
__global__ void __launch_bounds__(1024) scan_tile_offsets(double *bsum, long long nb, double *tot) {
    __shared__ double wsum[32];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const long long i0 = (long long)blockIdx.x * SCAN_TILE + 8LL * threadIdx.x;
    double v[8], a = 0.0;
#pragma unroll
    for (int k = 0; k < 8; ++k) {
        v[k] = i0 + k < nb ? bsum[i0 + k] : 0.0;
        a += v[k];
    }
    double s = a;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const double u = __shfl_up_sync(0xffffffffu, s, o);
        if (lane >= o) s += u;
    }
    if (lane == 31) wsum[warp] = s;
    __syncthreads();
    if (warp == 0) {
        double w = wsum[lane];
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const double u = __shfl_up_sync(0xffffffffu, w, o);
            if (lane >= o) w += u;
        }
        wsum[lane] = w;
    }
    __syncthreads();
    double run = (warp ? wsum[warp - 1] : 0.0) + (s - a);
#pragma unroll
    for (int k = 0; k < 8; ++k)
        if (i0 + k < nb) {
            bsum[i0 + k] = run;
            run += v[k];
        }
    if (threadIdx.x == 0) (gridDim.x == 1 ? bsum[nb] : tot[blockIdx.x]) = wsum[31];
}
// several tiles: add the totals of the tiles before each (at most 32: N = 30)
__global__ void __launch_bounds__(1024) scan_tile_add(double *bsum, long long nb, const double *tot) {
    double before = 0.0;
    for (unsigned g = 0; g < blockIdx.x; ++g) before += tot[g];
    const long long i0 = (long long)blockIdx.x * SCAN_TILE;
    for (long long i = i0 + threadIdx.x; i < i0 + SCAN_TILE && i < nb; i += 1024) bsum[i] += before;
    if (threadIdx.x == 0 && blockIdx.x == gridDim.x - 1) bsum[nb] = before + tot[blockIdx.x];
}

__global__ void __launch_bounds__(256) scan_chunk_apply(const double *p, unsigned long long n, const double *boff,
                                                        double *cdf) {
    __shared__ double part[257];
    const unsigned long long base = (unsigned long long)blockIdx.x * SCAN_CHUNK + threadIdx.x * 16ULL;
    double loc[16];
    double a = 0.0;
#pragma unroll
    for (int i = 0; i < 16; ++i) {
        loc[i] = (base + i < n) ? p[base + i] : 0.0;
        a += loc[i];
    }
    part[threadIdx.x + 1] = a;
    __syncthreads();
    if (threadIdx.x == 0) {
        part[0] = boff[blockIdx.x];
        for (int t = 1; t <= 256; ++t) part[t] += part[t - 1];
    }
    __syncthreads();
    double run = part[threadIdx.x];
#pragma unroll
    for (int i = 0; i < 16; ++i) {
        run += loc[i];
        if (base + i < n) cdf[base + i] = run;
    }
}

// chunk sums and their prefix; with cdf, the whole inclusive CDF as well
cudaError_t launch_scan(const double *p, unsigned long long n, double *cdf, double *bsum, double *tot,
                        int *launches, cudaStream_t st) {
    const long long nb = (long long)((n + SCAN_CHUNK - 1) / SCAN_CHUNK), tiles = (nb + SCAN_TILE - 1) / SCAN_TILE;
    scan_chunk_sums<<<(unsigned)nb, 256, 0, st>>>(p, n, bsum);
    scan_tile_offsets<<<(unsigned)tiles, 1024, 0, st>>>(bsum, nb, tot);
    if (tiles > 1) scan_tile_add<<<(unsigned)tiles, 1024, 0, st>>>(bsum, nb, tot);
    if (cdf) scan_chunk_apply<<<(unsigned)nb, 256, 0, st>>>(p, n, bsum, cdf);
    *launches = 2 + (tiles > 1 ? 1 : 0) + (cdf ? 1 : 0);
    return cudaGetLastError();
}

// ---------------------------------------------------------------- draws
// The smallest x with cdf[x] > t, or n - 1, and from there down to the last x of
// positive p: the prefixes round differently where threads, chunks and scan tiles
// meet, so the CDF may step at an x whose p is zero. Chunks whose sum did not move
// the prefix are passed over (boff as in launch_scan).
__device__ __forceinline__ unsigned long long cdf_search(const double *cdf, const double *p, const double *boff,
                                                         unsigned long long n, double t) {
    unsigned long long lo = 0, hi = n - 1;
    while (lo < hi) {
        const unsigned long long mid = lo + ((hi - lo) >> 1);
        if (cdf[mid] > t) hi = mid; else lo = mid + 1;
    }
    for (;;) {
        unsigned long long c = lo / SCAN_CHUNK;
        while (lo > c * SCAN_CHUNK && !(p[lo] > 0.0)) --lo;
        if (c == 0 || p[lo] > 0.0) return lo;
        do --c; while (c > 0 && !(boff[c + 1] > boff[c]));
        lo = (c + 1) * SCAN_CHUNK - 1;
    }
}

__global__ void draw_x_kernel(const double *cdf, const double *p, const double *boff, int N, long long n_x, int mode,
                              unsigned long long seed, unsigned long long ctr0, unsigned long long *xs) {
    const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n_x) return;
    const unsigned long long d = 1ULL << N;
    const double u = mc_uniform(seed, ctr0, (unsigned long long)i, 0ULL);
    unsigned long long x;
    if (i == 0) {
        x = 0ULL;          // x = 0 is its own stratum in both modes (SM Sec. I)
    } else if (mode == 0) {   // uniform on 1..d-1
        x = 1ULL + (unsigned long long)(u * (double)(d - 1));
        if (x >= d) x = d - 1;
    } else {                  // x ~ p(x | x != 0): inverse CDF over x >= 1
        const double c0 = cdf[0];
        x = cdf_search(cdf, p, boff, d, c0 + u * (cdf[d - 1] - c0));
        if (x == 0) x = 1;
    }
    xs[i] = x;
}

// x draws straight from p and the prefix of its chunk sums, without the CDF: a
// block per draw finds the chunk by bisection and sums that chunk alone. Family 0
// is x = 0; the others x ~ p(x | x != 0). Only x of positive p are drawn: the
// prefixes round where threads, chunks and scan tiles meet, so t may lie at or
// above the last sum (p(0) near 1 leaves few values between c0 and the total) or
// in a gap before a p of zero. The last positive p below is taken then, in the
// chunk or in the next lower one that holds any.
__global__ void __launch_bounds__(128) draw_x_chunk_kernel(const double *p, const double *boff, int N, long long nb,
                                                           unsigned long long seed, unsigned long long ctr0,
                                                           unsigned long long *xs) {
    __shared__ double wsum[4];
    __shared__ int first, last;            // of the chunk: the draw, and the last x of positive p
    __shared__ long long below;
    const long long i = blockIdx.x;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    if (i == 0) {
        if (threadIdx.x == 0) xs[0] = 0ULL;
        return;
    }
    const double c0 = p[0], total = boff[nb];
    const double t = c0 + mc_uniform(seed, ctr0, (unsigned long long)i, 0ULL) * (total - c0);
    long long lo = 0, hi = nb - 1;                 // smallest chunk whose end lies above t, else the last
    while (lo < hi) {
        const long long mid = (lo + hi) >> 1;
        if (boff[mid + 1] > t) hi = mid; else lo = mid + 1;
    }
    constexpr int CHUNK = (int)SCAN_CHUNK, PER = CHUNK / 128;
    for (;;) {
        const double *q = p + (unsigned long long)lo * CHUNK + (unsigned long long)threadIdx.x * PER;
        double v[PER], a = 0.0;
#pragma unroll
        for (int k = 0; k < PER; ++k) {
            v[k] = q[k];
            a += v[k];
        }
        double s = a;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const double u = __shfl_up_sync(0xffffffffu, s, o);
            if (lane >= o) s += u;
        }
        if (lane == 31) wsum[warp] = s;
        if (threadIdx.x == 0) { first = CHUNK; last = -1; below = 0; }
        __syncthreads();
        double run = boff[lo];
        for (int w = 0; w < warp; ++w) run += wsum[w];
        run += s - a;
        int pick = CHUNK, end = -1;
#pragma unroll
        for (int k = 0; k < PER; ++k) {
            run += v[k];
            if (v[k] > 0.0) {
                end = (int)threadIdx.x * PER + k;
                if (run > t && pick == CHUNK) pick = end;
            }
        }
        if (pick < CHUNK) atomicMin(&first, pick);
        if (end >= 0) atomicMax(&last, end);
        __syncthreads();
        const int f = first, l = last;
        if (f < CHUNK || l >= 0 || lo == 0) {
            if (threadIdx.x == 0) {
                const unsigned long long x = (unsigned long long)lo * CHUNK + (unsigned)(f < CHUNK ? f : l >= 0 ? l : 0);
                xs[i] = x ? x : 1ULL;
            }
            return;
        }
        // an empty chunk: the nearest one below whose sum moved the prefix, else chunk 0
        for (hi = lo; hi > 0; hi -= 128) {
            const long long c = hi - 1 - (long long)threadIdx.x;
            const bool up = c >= 0 && boff[c + 1] > boff[c];
            if (up) atomicMax((unsigned long long *)&below, (unsigned long long)c);
            if (__syncthreads_or(up)) break;
        }
        lo = below;
        __syncthreads();
    }
}

cudaError_t launch_draw_x_chunks(const double *p, const double *boff, int N, long long n_x, unsigned long long seed,
                                 unsigned long long ctr0, unsigned long long *xs, cudaStream_t st) {
    const long long nb = (long long)((1ULL << N) / SCAN_CHUNK);
    draw_x_chunk_kernel<<<(unsigned)n_x, 128, 0, st>>>(p, boff, N, nb, seed, ctr0, xs);
    return cudaGetLastError();
}

cudaError_t launch_draw_x(const double *cdf, const double *p, const double *boff, int N, long long n_x, int mode,
                          unsigned long long seed, unsigned long long ctr0, unsigned long long *xs, cudaStream_t st) {
    draw_x_kernel<<<(unsigned)((n_x + 255) / 256), 256, 0, st>>>(cdf, p, boff, N, n_x, mode, seed, ctr0, xs);
    return cudaGetLastError();
}

// z-range selection: the FP32 range weights Wf[f][.] -> their inclusive FP64
// scan W[f][.] (fixed order), then each draw k picks range r and the
// remainder t' within it.
// First level of the z draw for one family per CTA. Thread t owns the
// contiguous ranges [t per, (t + 1) per) ("chunk" t). The FP64 CDF is
// C(i) = S_t + (w_lo + ... + w_i) for i in chunk t, summed in range order from
// the chunk's start S_t, where S_t is the inclusive scan of the chunk sums
// (each chunk summed as four interleaved partial sums, the scan by warp
// shuffles: short FP64 dependency chains on a narrow FP64 pipe). Draw k picks
// the chunk a with S_a <= t < S_{a+1}, t = u_k S_256, then the smallest range
// r of it with C(r) > t; if rounding leaves C below t at the chunk's end (or t
// reaches the total), the last range of positive weight is taken and its
// remainder is clamped by the sampler. It records t - C(r - 1) and the
// range's weight C(r) - C(r - 1). Rows of at most ZSEL_STAGE_MAX ranges (a
// power of two) are first staged in shared memory by coalesced loads, with
// one padding word per chunk so the chunk-wise reads are free of bank
// conflicts.
__global__ void __launch_bounds__(256) zrange_select_kernel(const float *Wf, long long nr, long long n_fam,
                                                            long long fam_base, int z_per_x, unsigned long long seed,
                                                            unsigned long long ctr0, DrawInfo *draws,
                                                            const unsigned long long *perm) {
    __shared__ double seg[257];     // seg[t] = S_t, seg[256] = the total
    __shared__ double wsum[8];
    extern __shared__ float swf[];
    const long long f = blockIdx.x;
    if (f >= n_fam) return;
    // the family's own index: its draw stream and its draw records
    const unsigned long long fam = perm ? perm[fam_base + f] : (unsigned long long)(fam_base + f);
    const long long per = (nr + 255) / 256;
    const float *wrow = Wf + (size_t)f * nr;
    const int lp = 31 - __clz((int)per);
    for (uint32_t i = threadIdx.x; i < (uint32_t)nr; i += 256) swf[i + (i >> lp)] = wrow[i];
    __syncthreads();
    auto wf = [&](long long i) -> double { return (double)swf[(uint32_t)i + ((uint32_t)i >> lp)]; };
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const long long lo = tid * per, hi = lo + per < nr ? lo + per : nr;
    double a0 = 0.0, a1 = 0.0, a2 = 0.0, a3 = 0.0;
    long long i = lo;
    for (; i + 3 < hi; i += 4) {
        a0 += wf(i);
        a1 += wf(i + 1);
        a2 += wf(i + 2);
        a3 += wf(i + 3);
    }
    for (; i < hi; ++i) a0 += wf(i);
    double v = (a0 + a1) + (a2 + a3);
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const double u = __shfl_up_sync(0xffffffffu, v, o);
        if (lane >= o) v += u;
    }
    if (lane == 31) wsum[warp] = v;
    __syncthreads();
    if (warp == 0) {
        double w = lane < 8 ? wsum[lane] : 0.0;
#pragma unroll
        for (int o = 1; o < 8; o <<= 1) {
            const double u = __shfl_up_sync(0xffffffffu, w, o);
            if (lane >= o) w += u;
        }
        if (lane < 8) wsum[lane] = w;
    }
    __syncthreads();
    seg[tid + 1] = v + (warp > 0 ? wsum[warp - 1] : 0.0);
    if (tid == 0) seg[0] = 0.0;
    __syncthreads();
    const int tlast = (int)((nr - 1) / per);     // the last chunk that holds ranges
    const double total = seg[256];
    for (int k = tid; k < z_per_x; k += 256) {
        const double u = mc_uniform(seed, ctr0, fam, 1ULL + (unsigned long long)k);
        const double t = u * total;
        long long r = -1;
        double clo = 0.0, chi = 0.0;
        if (total > t) {
            int a = 0, b = tlast;                  // smallest a with S_{a+1} > t
            while (a < b) {
                const int mid = (a + b) >> 1;
                if (seg[mid + 1] > t) b = mid; else a = mid + 1;
            }
            const long long c0 = (long long)a * per, c1 = c0 + per < nr ? c0 + per : nr;
            double run = seg[a], lastp_lo = 0.0, lastp_hi = 0.0;
            long long lastp = -1;
            for (long long q = c0; q < c1; ++q) {
                const double w = wf(q), nrun = run + w;
                if (w > 0.0) { lastp = q; lastp_lo = run; lastp_hi = nrun; }
                if (nrun > t) { r = q; clo = run; chi = nrun; break; }
                run = nrun;
            }
            if (r < 0 && lastp >= 0) { r = lastp; clo = lastp_lo; chi = lastp_hi; }
        }
        if (r < 0) {
            // t at or past the total (or a chunk without weight): the last
            // range of positive weight
            for (int c = tlast; c >= 0 && r < 0; --c) {
                if (!(seg[c + 1] > seg[c])) continue;
                const long long c0 = (long long)c * per, c1 = c0 + per < nr ? c0 + per : nr;
                double run = seg[c];
                for (long long q = c0; q < c1; ++q) {
                    const double w = wf(q), nrun = run + w;
                    if (w > 0.0) { r = q; clo = run; chi = nrun; }
                    run = nrun;
                }
            }
            if (r < 0) { r = 0; clo = 0.0; chi = wf(0); }
        }
        DrawInfo di;
        di.range = (unsigned long long)r;
        di.t = t - clo;
        di.wr = chi - clo;
        di.pad = 0.0;
        draws[(size_t)fam * z_per_x + k] = di;
    }
}

// The same selection for rows of more than ZSEL_STAGE_MAX ranges, in two launches
// that add in the same order: a thread of zrange_select_kernel walked its chunk
// (4096 ranges at N = 30) through uncached loads, 1.33 ms for 8 families; these
// take 0.12 + 0.27 ms (chains of dependent FP64 additions).
// zchunk_sums_kernel: lane (chunk, chain q) adds the ranges 4 i + q of the chunk.
__global__ void __launch_bounds__(32) zchunk_sums_kernel(const float *Wf, long long nr, double *sums) {
    const long long per = nr / 256;
    const int lane = threadIdx.x, q = lane & 3;
    const long long chunk = 8LL * blockIdx.x + (lane >> 2);
    const float *w = Wf + (size_t)blockIdx.y * nr + chunk * per + q;
    double a = 0.0;
    for (long long i = 0; i < per; i += 64) {          // per is a power of two, at least 128
        float v[16];
#pragma unroll
        for (int k = 0; k < 16; ++k) v[k] = w[i + 4 * k];
#pragma unroll
        for (int k = 0; k < 16; ++k) a += f2d(v[k]);
    }
    // (a0 + a1) + (a2 + a3)
    a += __shfl_xor_sync(0xffffffffu, a, 1);
    a += __shfl_xor_sync(0xffffffffu, a, 2);
    if (q == 0) sums[256 * (size_t)blockIdx.y + chunk] = a;
}
// A block per family and ZSEL_DRAWS draws, a warp per draw: the chunk's ranges
// arrive 32 at a time and are added one after another.
constexpr int ZSEL_DRAWS = 4;
__global__ void __launch_bounds__(32 * ZSEL_DRAWS) zrange_draw_kernel(const float *Wf, long long nr, const double *sums,
                                                                      long long fam_base, int z_per_x,
                                                                      unsigned long long seed, unsigned long long ctr0,
                                                                      DrawInfo *draws, const unsigned long long *perm) {
    __shared__ double seg[257];
    const long long f = blockIdx.y;
    const unsigned long long fam = perm ? perm[fam_base + f] : (unsigned long long)(fam_base + f);
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const float *wrow = Wf + (size_t)f * nr;
    const long long per = nr / 256;
    if (warp == 0) {
        // the scan of zrange_select_kernel: warps of 32 chunks, then their sums
        double wv[8], ws = 0.0;
#pragma unroll
        for (int w = 0; w < 8; ++w) {
            double v = sums[256 * (size_t)f + 32 * w + lane];
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const double u = __shfl_up_sync(0xffffffffu, v, o);
                if (lane >= o) v += u;
            }
            wv[w] = v;
            const double last = __shfl_sync(0xffffffffu, v, 31);
            if (lane == w) ws = last;
        }
#pragma unroll
        for (int o = 1; o < 8; o <<= 1) {
            const double u = __shfl_up_sync(0xffffffffu, ws, o);
            if (lane >= o) ws += u;
        }
#pragma unroll
        for (int w = 0; w < 8; ++w) {
            const double before = __shfl_sync(0xffffffffu, ws, w > 0 ? w - 1 : 0);
            seg[1 + 32 * w + lane] = wv[w] + (w > 0 ? before : 0.0);
        }
        if (lane == 0) seg[0] = 0.0;
    }
    __syncthreads();
    const int k = blockIdx.x * ZSEL_DRAWS + warp;
    if (k >= z_per_x) return;
    const double total = seg[256];
    const double t = mc_uniform(seed, ctr0, fam, 1ULL + (unsigned long long)k) * total;
    long long r = -1;
    double clo = 0.0, chi = 0.0;
    // walk one chunk from its start; the first range whose end lies above tt,
    // else (or for tt = infinity) the last one of positive weight
    auto walk = [&](int chunk, double tt) {
        const long long c0 = (long long)chunk * per;
        double run = seg[chunk];
        float next = wrow[c0 + lane];
        for (long long b = 0; b < per; b += 32) {
            const double w = f2d(next);
            if (b + 32 < per) next = wrow[c0 + b + 32 + lane];
            // every lane adds all 32 in turn; lane i keeps the sums around its range
            double before = 0.0, after = 0.0;
#pragma unroll
            for (int i = 0; i < 32; ++i) {
                const double nrun = run + __shfl_sync(0xffffffffu, w, i);
                before = i == lane ? run : before;
                after = i == lane ? nrun : after;
                run = nrun;
            }
            const unsigned hits = __ballot_sync(0xffffffffu, after > tt);
            const unsigned pos = __ballot_sync(0xffffffffu, w > 0.0);
            // a hit ends the walk; otherwise remember the last range of positive weight
            const int pick = hits ? __ffs(hits) - 1 : 31 - __clz(pos);
            if (pick >= 0) {
                r = c0 + b + pick;
                clo = __shfl_sync(0xffffffffu, before, pick);
                chi = __shfl_sync(0xffffffffu, after, pick);
            }
            if (hits) break;
        }
    };
    if (total > t) {
        int a = 0, b = 255;                            // smallest a with S_{a+1} > t
        while (a < b) {
            const int mid = (a + b) >> 1;
            if (seg[mid + 1] > t) b = mid; else a = mid + 1;
        }
        walk(a, t);
    }
    if (r < 0)
        for (int c = 255; c >= 0 && r < 0; --c)
            if (seg[c + 1] > seg[c]) walk(c, __longlong_as_double(0x7ff0000000000000LL));
    if (r < 0) { r = 0; clo = 0.0; chi = (double)wrow[0]; }
    if (lane == 0) {
        DrawInfo di;
        di.range = (unsigned long long)r;
        di.t = t - clo;
        di.wr = chi - clo;
        di.pad = 0.0;
        draws[(size_t)fam * z_per_x + k] = di;
    }
}

cudaError_t launch_zrange_select(const float *Wf, long long nr, long long n_fam, long long fam_base, int z_per_x,
                                 unsigned long long seed, unsigned long long ctr0, DrawInfo *draws,
                                 const unsigned long long *perm, double *sums, int *launches, cudaStream_t st) {
    if (nr & (nr - 1)) return cudaErrorInvalidValue;         // 2^(N - RL)
    if (nr <= ZSEL_STAGE_MAX) {
        const size_t smem = sizeof(float) * (size_t)(nr + 256 + 1);
        static SmemOptIn optin;
        const cudaError_t e = optin.allow((const void *)zrange_select_kernel, sizeof(float) * (ZSEL_STAGE_MAX + 257));
        if (e != cudaSuccess) return e;
        zrange_select_kernel<<<(unsigned)n_fam, 256, smem, st>>>(Wf, nr, n_fam, fam_base, z_per_x, seed, ctr0, draws,
                                                                 perm);
        *launches = 1;
        return cudaGetLastError();
    }
    // at most 128 families a launch here (N >= 25)
    zchunk_sums_kernel<<<dim3(32, (unsigned)n_fam), 32, 0, st>>>(Wf, nr, sums);
    zrange_draw_kernel<<<dim3((unsigned)((z_per_x + ZSEL_DRAWS - 1) / ZSEL_DRAWS), (unsigned)n_fam), 32 * ZSEL_DRAWS, 0, st>>>(
        Wf, nr, sums, fam_base, z_per_x, seed, ctr0, draws, perm);
    *launches = 2;
    return cudaGetLastError();
}

// ------------------------------------------------------------ MC statistics
// Per family i: y[i][0..2] = mean over its z-draws of (-log2 c^2, c^2, c^4);
// y[i][3..5] = the family's exact conditional means (-sum c^2 log2 c^2,
// sum c^4, sum c^6) / sum c^2 (marginal mode; family 0, the x = 0 stratum,
// takes the exact means in both slots), or, uniform mode, the SM Sec. I
// family values h_x, m_{2;x}, m_{3;x} in y[i][0..2]. A warp per family, lanes over
// its draws (a thread per family
// left most SMs idle: N = 24, 4096 families of 256 draws 240 us, now 52 us)
__global__ void __launch_bounds__(256) mc_family_stats_kernel(const FamMoments *fm, const float *cz, long long n_x,
                                                              int z_per_x, int N, int mode, double *y) {
    const int lane = threadIdx.x & 31;
    const long long i = (long long)blockIdx.x * 8 + (threadIdx.x >> 5);
    if (i >= n_x) return;
    const double d = ldexp(1.0, N);
    const FamMoments m = fm[i];
    double *o = y + 6 * i;
    if (mode == 0) {
        if (lane == 0) {
            o[0] = N * (m.m[0] / d) - m.m[3] / d;
            o[1] = m.m[1] / (d * d);
            o[2] = m.m[2] / (d * d * d);
            o[3] = o[4] = o[5] = 0.0;
        }
        return;
    }
    double a[4] = {0.0, 0.0, 0.0, 0.0};
    if (i > 0)
        for (int k = lane; k < z_per_x; k += 32) {
            const double c = (double)cz[(size_t)i * z_per_x + k];
            const double c2 = c * c;
            a[0] += -log2(c2);
            a[1] += c2;
            a[2] += c2 * c2;
        }
    int id;
    const double t = warp_sums<4>(a, id);                // value v in lanes 8 v .. 8 v + 7
    if ((lane & 7) == 0 && id < 3) {
        // p(x) may be the marginal's rounding alone (below 2^-50 or so of p(0)): a
        // drawn family whose c are all zero has no conditional means and adds nothing
        const bool none = m.m[0] == 0.0;
        const double exact = none ? 0.0 : (id == 0 ? -m.m[3] : id == 1 ? m.m[1] : m.m[2]) / m.m[0];
        o[3 + id] = exact;
        o[id] = i == 0 ? exact : none ? 0.0 : t / z_per_x;
    }
}

// out[0..5] = sum_{i >= first} y[i][a], out[6..11] = sum y^2, out[12..17] = y[0][a],
// out[18] = sum over families of sum c^2 / (d p(x)) estimate (marginal) -- fixed
// order, one block per value (one block for all: 165 us for 5001 families).
__global__ void __launch_bounds__(256) mc_totals_kernel(const double *y, long long n_x, int first,
                                                        const FamMoments *fm, double *out) {
    __shared__ double red[8];
    const int a = blockIdx.x;
    NeuSum ns, nq;
    if (a < 6) {
        for (long long i = first + threadIdx.x; i < n_x; i += 256) {
            const double v = y[6 * i + a];
            ns.add(v);
            nq.add(v * v);
        }
    } else {
        for (long long i = threadIdx.x; i < n_x; i += 256) ns.add(fm[i].m[0]);
    }
    const double s = block_sum<256>(ns.value(), red);
    if (a == 6) {
        if (threadIdx.x == 0) out[18] = s;
        return;
    }
    const double q = block_sum<256>(nq.value(), red);
    if (threadIdx.x == 0) { out[a] = s; out[6 + a] = q; out[12 + a] = y[a]; }
}

cudaError_t launch_mc_stats(const FamMoments *fm, const float *cz, long long n_x, int z_per_x, int N, int mode,
                            double *y, double *out, cudaStream_t st) {
    mc_family_stats_kernel<<<(unsigned)((n_x + 7) / 8), 256, 0, st>>>(fm, cz, n_x, z_per_x, N, mode, y);
    mc_totals_kernel<<<7, 256, 0, st>>>(y, n_x, 1, fm, out);
    return cudaGetLastError();
}

// ------------------------------------------------------- batched states
// per-state sum |psi|^2: grid (blocks per state, states), fixed order
__global__ void __launch_bounds__(256) norm2_multi_partial(const float2 *const *psi_list, int N, int nb,
                                                           double *partial) {
    __shared__ double red[8];
    const int st = blockIdx.y;
    const double acc = block_sum<256>(norm2_part(psi_list[st], 1ULL << N, (unsigned long long)blockIdx.x * 256 + threadIdx.x,
                                                 (unsigned long long)nb * 256), red);
    if (threadIdx.x == 0) partial[(size_t)st * nb + blockIdx.x] = acc;
}

__global__ void __launch_bounds__(256) norm2_multi_final(const double *partial, int nb, double *norm2, double *s) {
    __shared__ double red[8];
    const int st = blockIdx.x;
    double acc = 0.0;
    for (int i = threadIdx.x; i < nb; i += 256) acc += partial[(size_t)st * nb + i];
    acc = block_sum<256>(acc, red);
    if (threadIdx.x == 0) {
        norm2[st] = acc;
        s[st] = acc > 0.0 ? 1.0 / acc : 0.0;
    }
}

cudaError_t launch_norm2_multi(const float2 *const *psi_list, int n_states, int N, double *partial, int nb,
                               double *norm2, double *s, cudaStream_t st) {
    norm2_multi_partial<<<dim3(nb, n_states), 256, 0, st>>>(psi_list, N, nb, partial);
    norm2_multi_final<<<n_states, 256, 0, st>>>(partial, nb, norm2, s);
    return cudaGetLastError();
}

// stab counts of flagged families added to their states (integer atomics)
__global__ void count_scatter_kernel(const unsigned long long *flags, const unsigned long long *counts, long long n,
                                     int N, unsigned long long *state_count) {
    const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    if (counts[i]) atomicAdd(state_count + (flags[i] >> N), counts[i]);
}

cudaError_t launch_count_scatter(const unsigned long long *flags, const unsigned long long *counts, long long n,
                                 int N, unsigned long long *state_count, cudaStream_t st) {
    if (n <= 0) return cudaSuccess;
    count_scatter_kernel<<<(unsigned)((n + 255) / 256), 256, 0, st>>>(flags, counts, n, N, state_count);
    return cudaGetLastError();
}

cudaError_t launch_philox_test(const unsigned long long *ctr_key, unsigned long long *out, int n, cudaStream_t st) {
    philox_test_kernel<<<(n + 127) / 128, 128, 0, st>>>(ctr_key, out, n);
    return cudaGetLastError();
}

} // namespace sre
