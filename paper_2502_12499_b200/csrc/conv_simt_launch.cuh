// Instantiations of the CUDA-core convolution for one storage type (included by one translation unit per type).
#pragma once
#include "conv_simt.cuh"

namespace ckpt {
namespace simt {

template <typename T, int MODE, int BM, int BN, int TM, int TN, bool VA, bool VB, Form FORM = Form::CHAINS>
static int go(const ConvGeom& g, const void* a, const void* b, void* out, const float* bias, int relu, int M, int N, int K, const Plan& p,
              const SgdUpdate& upd, cudaStream_t st, float* sums) {
    using L = Tile<T, MODE, BM, BN, TM, TN>;
    auto kernel = conv_gemm_kernel<T, MODE, BM, BN, TM, TN, VA, VB, FORM>;
    if (L::smem > 48 * 1024) {
        static DeviceFlags ready;
        if (int bad = allow_shared_memory(ready, {(const void*)kernel}, L::smem)) return bad;
    }
    cudaLaunchConfig_t cfg = {};
    unsigned m_tiles = (unsigned)((M + BM - 1) / BM);
    if (MODE == 1 && g.stride > 1) {        // one set of tiles per parity class of the input, sized for the largest class
        const int64_t px = (int64_t)g.n * ((g.h + g.stride - 1) / g.stride) * ((g.w + g.stride - 1) / g.stride);
        m_tiles = (unsigned)((px + BM - 1) / BM) * (unsigned)(g.stride * g.stride);
    }
    cfg.gridDim = dim3(m_tiles, (unsigned)((N + BN - 1) / BN), (unsigned)(p.slices * p.cluster));
    cfg.blockDim = dim3(L::threads);
    cfg.dynamicSmemBytes = L::smem;
    cfg.stream = st;
    cudaLaunchAttribute attr[2];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = 1; attr[0].val.clusterDim.y = 1; attr[0].val.clusterDim.z = (unsigned)p.cluster;
    cfg.attrs = attr;
    cfg.numAttrs = p.cluster > 1 ? 1 : 0;
    start_early(&cfg, attr, Start::ON_STREAMS);
    cudaError_t e = cudaLaunchKernelEx(&cfg, kernel, g, (const T*)a, (const T*)b, out, bias, relu, M, N, K, p.k_per_slice, p.cluster, upd, sums);
    if (e != cudaSuccess) return cuda_fail(e, "launching the CUDA-core convolution");
    static const char* const names[3] = {"conv forward (CUDA cores)", "conv dgrad (CUDA cores)", "conv wgrad (CUDA cores)"};
    CKPT_LAUNCH_CHECK_NAMED(names[MODE], names[MODE]);
    return CKPT_OK;
}

// 16-byte chunks: every tile shape, through a filter of more than 16 rows the four that won any; value by value: three (see plan)
template <typename T, int MODE, bool VA, bool VB>
static int pick(const ConvGeom& g, const void* a, const void* b, void* out, const float* bias, int relu, int M, int N, int K, const Plan& p,
                const SgdUpdate& upd, cudaStream_t st, float* sums) {
    const bool one = MODE != 2 && !VA && !VB && p.k_per_slice <= kChain && (p.tile == 2 || p.tile == 4 || p.tile == 6);
#define CKPT_CASE(I, BM, BN, TM, TN)                                                                                   \
    if constexpr ((VA && VB) || I == 2 || I == 4 || I == 6)                                                            \
        if (p.tile == I && !p.wide && !one) return go<T, MODE, BM, BN, TM, TN, VA, VB>(g, a, b, out, bias, relu, M, N, K, p, upd, st, sums);    \
    if constexpr (MODE != 2 && VA && (I == 2 || (VB && I == 3) || I == 4 || I == 6))                                   \
        if (p.tile == I && p.wide) return go<T, MODE, BM, BN, TM, TN, VA, VB, Form::WIDE>(g, a, b, out, bias, relu, M, N, K, p, upd, st, sums);    \
    if constexpr (MODE != 2 && !VA && !VB && (I == 2 || I == 4 || I == 6))                                              \
        if (p.tile == I && one) return go<T, MODE, BM, BN, TM, TN, VA, VB, Form::ONE_CHAIN>(g, a, b, out, bias, relu, M, N, K, p, upd, st, sums);
    if constexpr (MODE == 2) { CKPT_SIMT_TILES_W(CKPT_CASE) } else { CKPT_SIMT_TILES(CKPT_CASE) }
#undef CKPT_CASE
    set_error("CUDA-core convolution: no such tile");
    return CKPT_E_UNSUPPORTED;
}

template <typename T>
int launch(int mode, const ConvGeom& g, const void* a, const void* b, void* out, const float* bias, int relu, int M, int N, int K,
           bool va, bool vb, const Plan& p, const SgdUpdate& upd, cudaStream_t st, float* sums) {
    if (mode == 0)      // both operands run along the input channels
        return va && vb ? pick<T, 0, true, true>(g, a, b, out, bias, relu, M, N, K, p, upd, st, sums) : pick<T, 0, false, false>(g, a, b, out, bias, relu, M, N, K, p, upd, st, sums);
#define CKPT_MODE(MODE)                                                                                                \
    if (va && vb) return pick<T, MODE, true, true>(g, a, b, out, bias, relu, M, N, K, p, upd, st, sums);                          \
    if (va) return pick<T, MODE, true, false>(g, a, b, out, bias, relu, M, N, K, p, upd, st, sums);                               \
    if (vb) return pick<T, MODE, false, true>(g, a, b, out, bias, relu, M, N, K, p, upd, st, sums);                               \
    return pick<T, MODE, false, false>(g, a, b, out, bias, relu, M, N, K, p, upd, st, sums);
    if (mode == 1) { CKPT_MODE(1) }
    CKPT_MODE(2)
#undef CKPT_MODE
}

}  // namespace simt
}  // namespace ckpt
