// Instantiations: FP32 strided passes (2^K rows x 2^(MS-K) columns) and row passes.
#include "k_pass_dispatch.cuh"
namespace sre {
namespace {
// six bits in one round of 64 points per thread; the split-BF16 form keeps 32
template <int SRC>
cudaError_t strided6(const PassArgs &a, int tiles, cudaStream_t st) {
    constexpr int M = f32_strided_ms(6);
    if (a.precision == 0) return launch_cfg<TileCfg<float, M, M - 6, 6, 1>, SRC, DST_BUF, 0>(a, tiles, st);
    if (a.precision == 2) return launch_cfg<TileCfg<float, M, M - 6, 5, 1>, SRC, DST_BUF, 2>(a, tiles, st);
    if (a.precision == 3) return launch_cfg<TileCfg<float, M, M - 6, 5, 1>, SRC, DST_BUF, 3>(a, tiles, st);
    return cudaErrorInvalidValue;
}
} // namespace

cudaError_t launch_f32_strided(int MS, int K, int src, int dst, const PassArgs &a, int tiles, cudaStream_t st) {
    if (K == 10 && src == SRC_PSI_FAMILY && dst == DST_BUF && a.precision == 0 && a.psi_tiled && !a.psi_list)
        return launch_cfg<TileCfg<float, f32_strided_ms(10), PSI_TILED_COLS, f32_strided_rb(10), 1>, SRC_PSI_TILED, DST_BUF, 0>(
            a, tiles, st);
    if (MS != f32_strided_ms(K)) {
        if (src != SRC_PSI_FAMILY || dst != DST_BUF || MS != f32_strided_ms(K, true)) return cudaErrorInvalidValue;
        switch (K) {
#define C(k) case k: return launch_if<KIND_STRIDED, TileCfg<float, f32_strided_ms(k, true), f32_strided_ms(k, true) - k, 5, 1>, SRC_PSI_FAMILY, DST_BUF>(a, tiles, st);
        C(7) C(8)
#undef C
        default: return cudaErrorInvalidValue;
        }
    }
    switch (K) {
#define C(k) case k: return launch_sd<KIND_STRIDED, TileCfg<float, f32_strided_ms(k), f32_strided_ms(k) - k, f32_strided_rb(k), 1>>(src, dst, a, tiles, st);
    C(1) C(2) C(3) C(4) C(5) C(7) C(8) C(9) C(10)
#undef C
    case 6:
        if (dst != DST_BUF) return cudaErrorInvalidValue;
        if (src == SRC_PSI_FAMILY) return strided6<SRC_PSI_FAMILY>(a, tiles, st);
        if (src == SRC_BUF) return strided6<SRC_BUF>(a, tiles, st);
        return cudaErrorInvalidValue;
    default: return cudaErrorInvalidValue;
    }
}
cudaError_t launch_f32_row(int M, int src, int dst, const PassArgs &a, int tiles, cudaStream_t st) {
    // moments without z-range weights over 12 bits: 64 points per thread, one
    // exchange through shared memory instead of two (uniform sweep of N = 18,
    // per point: 1.46 against 1.78 ps; over 11 bits 1.65 against 1.64). Its FP32
    // sums cover no more than in the 32-point rows: chains of 32 points, FP64 from
    // 1024 points on (one chain of 64 and 2048 points: 1.44 ps, but up to 15 last
    // places off where 32 equal terms lose nothing)
    if (M == 12 && a.precision == 0 && src == SRC_BUF && dst == DST_MOMENTS && !a.want_ranges)
        return launch_cfg<TileCfg<float, 12, 0, 6, 1>, SRC_BUF, DST_MOMENTS, 0>(a, tiles, st);
    switch (M) {
#define C(m) case m: return launch_sd<KIND_ROW, TileCfg<float, m, 0, (m == 13 ? F32_ROW13_RB : 5), 1>>(src, dst, a, tiles, st);
    C(10) C(11) C(12) C(13) C(14)
#undef C
    default: return cudaErrorInvalidValue;
    }
}
} // namespace sre

namespace sre {
namespace {
// The 10-bit strided pass reads psi in 64-byte rows: a warp's 8-byte loads touch
// four half-used lines, and the tag stage of L1 bounded the pass (71% busy, loads
// throttled). From a copy of psi in which a tile's rows are contiguous, every load
// of a warp is two full lines: N = 24, 128 families per launch 2.79 -> 2.49 ms,
// 2.6 -> 2.3 ps per point (1.2 ps is the DRAM time of what it writes; its 64-byte
// stores are what is left); the step of 4096 families 172.7 -> 162.9 ms with the
// copy. psi in tile order: a thread per amplitude in the order of the copy, so that
// writes are contiguous and reads are the copy's 64-byte rows
__global__ void __launch_bounds__(256) psi_tile_kernel(const float2 *psi, float2 *out, int lo, int N) {
    constexpr int C = PSI_TILED_COLS, PER = 8;
    const uint32_t p0 = blockIdx.x * (256u * PER) + threadIdx.x;
    float2 v[PER];
#pragma unroll
    for (int i = 0; i < PER; ++i) {
        const uint32_t p = p0 + 256u * i;
        const uint32_t row = (p >> C) & ((1u << (N - lo)) - 1u), cb = p >> (N - lo + C);
        v[i] = __ldg(psi + ((p & ((1u << C) - 1u)) | (cb << C) | (row << lo)));
    }
#pragma unroll
    for (int i = 0; i < PER; ++i) out[p0 + 256u * i] = v[i];
}
} // namespace

cudaError_t launch_psi_tiled(const float2 *psi, float2 *out, int lo, int N, cudaStream_t st) {
    if (N < 11 || N > 31 || lo <= PSI_TILED_COLS || lo >= N) return cudaErrorInvalidValue;
    psi_tile_kernel<<<1u << (N - 11), 256, 0, st>>>(psi, out, lo, N);
    return cudaGetLastError();
}
} // namespace sre
