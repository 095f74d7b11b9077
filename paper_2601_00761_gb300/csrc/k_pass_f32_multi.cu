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
    // moments without z-range weights over 11 and 12 bits: 64 points per
    // thread, one exchange through shared memory instead of two (per point,
    // 4096 families of N = 18: 1.49 and 1.53 ps against 1.66 and 1.81)
    if ((M == 11 || M == 12) && a.precision == 0 && src == SRC_BUF && dst == DST_MOMENTS && !a.want_ranges)
        return M == 11 ? launch_cfg<TileCfg<float, 11, 0, 6, 1>, SRC_BUF, DST_MOMENTS, 0>(a, tiles, st)
                       : launch_cfg<TileCfg<float, 12, 0, 6, 1>, SRC_BUF, DST_MOMENTS, 0>(a, tiles, st);
    switch (M) {
#define C(m) case m: return launch_sd<KIND_ROW, TileCfg<float, m, 0, (m == 13 ? F32_ROW13_RB : 5), 1>>(src, dst, a, tiles, st);
    C(10) C(11) C(12) C(13) C(14)
#undef C
    default: return cudaErrorInvalidValue;
    }
}
} // namespace sre
