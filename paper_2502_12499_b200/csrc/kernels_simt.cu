// CUDA-core kernels: general implicit-GEMM convolution (forward, dgrad, wgrad; any filter size,
// stride, padding and channel count; float32 or bfloat16 storage with float32 accumulation),
// batch normalisation, pooling, losses and small element-wise helpers.
//
// Every reduction has a fixed summation order (no floating-point atomics), so repeated runs and
// recomputation give bit-identical results.
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstdint>
#include <cstdio>

#include "conv_simt.cuh"
#include "internal.h"
#include "overlap.cuh"
#include "vec.cuh"

namespace ckpt {

int cuda_fail(int err, const char* what) {
    set_error("CUDA error during %s: %s", what, cudaGetErrorString((cudaError_t)err));
    return CKPT_E_CUDA;
}

int allow_shared_memory(DeviceFlags& flags, std::initializer_list<const void*> kernels, int bytes) {
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return cuda_fail(e, "asking for the device");
    return flags.once(dev, [&] {
        for (const void* kernel : kernels)
            if ((e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes)) != cudaSuccess) return cuda_fail(e, "raising the shared-memory limit");
        return (int)CKPT_OK;
    });
}

ConvGeom make_geom(const ckpt_conv_shape& s) {
    ConvGeom g;
    g.n = s.n; g.h = s.h; g.w = s.w; g.cin = s.c_in; g.cout = s.c_out; g.k = s.k; g.stride = s.stride; g.pad = s.pad;
    g.ho = (s.h + 2 * s.pad - s.k) / s.stride + 1;
    g.wo = (s.w + 2 * s.pad - s.k) / s.stride + 1;
    return g;
}


// ================================================================================================
// Convolutions on the CUDA cores (kernel and tile shapes: conv_simt.cuh)
// ================================================================================================
namespace simt {
// The tile shape, the CTAs of a cluster that share a tile's reduction and (wgrad) the slices whose partial sums a second
// kernel adds: the cheapest by a model of clocks per SM.  148 SMs are written in: the scratch size of a chain comes from
// here and must not depend on the device at hand.
//
// Operands in 16-byte chunks: an SM holds `held` CTAs of a tile shape at once (the number that its kernel is compiled for) and works
// them off in rounds.  n of them need, per step along K, n times the tile's FMAs at the share of the peak that the shape reaches, and
// a wait that they spend once together.  The CTAs of a cluster share a GPC, which leaves some SMs short: clusters reach fewer of
// them (without that the choice is 3.0 % behind the best of a layer's plans in the mean, float32 forward of 62 layers, so 2.1).
// Fitted for each type to some 17,000 measured plans of 104 layers, each within 5-9 % on average; the chosen plan is 0.9-1.9 % behind
// the best of its layer in the mean, for bfloat16 1.1-2.9 (2.4-6.2 with float32's figures for both).
// us, float32, forward / dgrad / wgrad, one share per shape and no view of how many CTAs an SM holds -> this: 128 -> 128 at 8 x 8,
// 32 images 51/52/36 -> 29/28/22, 256 -> 256 3x3 stride 2 at 28 x 28, 16 images 165/320/148 -> 125/206/100, 1x1 64 -> 256 at 56 x 56, 8 images
// 33/39/63 -> 31/32/42.
struct TileShape { int m, n, held[2], held_values[2]; };         // held: float32, bfloat16
#define CKPT_SHAPE(MODE, BM, BN, TM, TN)                                                                                     \
    {BM, BN, {Tile<float, MODE, BM, BN, TM, TN>::held, Tile<__nv_bfloat16, MODE, BM, BN, TM, TN>::held},                     \
     {Tile<float, MODE, BM, BN, TM, TN>::held_values, Tile<__nv_bfloat16, MODE, BM, BN, TM, TN>::held_values}},
#define CKPT_SHAPE0(I, BM, BN, TM, TN) CKPT_SHAPE(0, BM, BN, TM, TN)
#define CKPT_SHAPE1(I, BM, BN, TM, TN) CKPT_SHAPE(1, BM, BN, TM, TN)
#define CKPT_SHAPE2(I, BM, BN, TM, TN) CKPT_SHAPE(2, BM, BN, TM, TN)
static constexpr TileShape kShapes[3][7] = {{CKPT_SIMT_TILES(CKPT_SHAPE0)}, {CKPT_SIMT_TILES(CKPT_SHAPE1)}, {CKPT_SIMT_TILES_W(CKPT_SHAPE2)}};
#undef CKPT_SHAPE
#undef CKPT_SHAPE0
#undef CKPT_SHAPE1
#undef CKPT_SHAPE2
struct TileCost { double share, wait; };
struct ModeCost { TileCost tile[7]; double round, exchange, exchange_tile, slice_sum, slice_share; };
static const ModeCost kCost[2][3] = {            // float32, bfloat16; modes
    {{{{0.47, 40}, {0.66, 70}, {0.67, 55}, {0.62, 65}, {0.54, 44}, {0.43, 39}, {0.41, 32}}, 2150, 2000, 21.7, 0, 0},
     {{{0.45, 40}, {0.65, 86}, {0.66, 67}, {0.62, 69}, {0.63, 44}, {0.52, 59}, {0.44, 33}}, 2390, 1730, 21.8, 0, 0},
     {{{0.63, 11}, {0.91, 98}, {0.82, 51}, {0.78, 77}, {0.73, 47}, {0.69, 73}, {0.48, 46}}, 40, 2700, 17.2, 2470, 0.91}},
    {{{{0.65, 26}, {0.92, 76}, {0.72, 49}, {0.65, 50}, {0.68, 35}, {0.68, 44}, {0.45, 19}}, 1410, 1850, 29.0, 0, 0},
     {{{0.49, 14}, {0.63, 70}, {0.86, 64}, {0.66, 52}, {0.73, 40}, {0.61, 42}, {0.45, 20}}, 870, 2000, 28.8, 0, 0},
     {{{0.60, 10}, {0.79, 65}, {0.72, 39}, {0.55, 42}, {0.57, 25}, {0.51, 34}, {0.41, 21}}, 40, 2550, 16.4, 2300, 0.84}}};
static int sms_in_reach(int cluster) { return 148 - (cluster > 1 ? 3 * cluster / 2 : 0); }
static int per_sm(int64_t ctas, int sms) { return (int)((ctas + sms - 1) / sms); }      // (whole numbers throughout: a chain's creation runs this some thousand times)
static double clocks_of_chunks(int mode, int value_bytes, int t, int64_t ctas, int per, int cluster, int slices, double outputs) {
    const ModeCost& c = kCost[value_bytes == 2][mode];
    const TileShape& s = kShapes[mode][t];
    const int held = s.held[value_bytes == 2];
    const int load = per_sm(ctas, sms_in_reach(cluster)), rounds = load / held, rest = load % held;
    const double fma = (double)s.m * s.n / 128.0 / c.tile[t].share;
    double clk = rounds * (per * (fma * held + c.tile[t].wait) + c.round);
    if (rest > 0) clk += per * (fma * rest + c.tile[t].wait) + c.round;
    if (cluster == 2 && load <= 2) clk *= 1.1;                // (a pair may come to share an SM while others have none: 9-16 % more, measured)
    if (cluster > 1) clk += c.exchange + load * c.exchange_tile * s.m * s.n / 32.0;
    if (slices > 1) clk += c.slice_sum + c.slice_share * slices * outputs * 8.0 / 2500.0;
    return clk;
}
// Operands fetched value by value: FMA time is the tile volume over 128 lanes and the share of the peak a tile shape reaches; a
// cluster costs its exchange, further slices a launch and a pass over the partial sums.  Such a weight gradient takes a CTA some
// 2200 clocks per step of 16 whatever its tile - four warps do not hide their addresses and reads - so that its long reduction
// wants more CTAs, also such a number of slices as rounds to fewer (us, 3 -> 256, 28 images of 13 x 49 float32 87 -> 34,
// 5 -> 20 at 28 x 28 69 -> 16, 3 -> 64 1x1 at 40 x 40, 20 images 67 -> 18, bfloat16 65 -> 21) - as many as an SM holds, or the steps
// count for each round of the grid (7x7 stride 2 3 -> 64 at 200 x 168, 21 images 213 -> 150).
static double clocks_of_values(int mode, int value_bytes, int t, int bm, int bn, int64_t ctas, int per, int cluster, int slices, double outputs) {
    static const double share[7] = {0.85, 0.8, 0.7, 0.6, 0.5, 0.4, 0.35};
    // CTAs per SM; one or two of 128 threads do not hide the latency of their shared-memory reads
    const int load = per_sm(ctas, 148);
    const double hidden = load < 2 ? 0.6 : load < 3 ? 0.8 : 1.0;
    double clk = load * ((double)bm * bn * per / (128.0 * share[t] * hidden) + 300.0);
    if (mode == 2) clk = std::max(clk, 140.0 * per * per_sm(per_sm(ctas, sms_in_reach(cluster)), kShapes[mode][t].held_values[value_bytes == 2]));
    clk += 2000.0;
    if (cluster > 1) clk += 1000.0 + load * bm * bn / 32.0;
    if (slices > 1) clk += 4000.0 + (double)slices * outputs * 8.0 / 2500.0;
    return clk;
}
Plan plan(int mode, int value_bytes, int M, int N, int K, bool vectors, bool wide) {
    Plan best{2, 1, 1, K, wide};
    double best_t = 1e300;
    for (int t = 0; t < 7; ++t) {
        if ((!vectors || wide) && t != 2 && t != 4 && t != 6 && !(vectors && t == 3)) continue;
        const int bm = kShapes[mode][t].m, bn = kShapes[mode][t].n;
        const int64_t tiles = (int64_t)((M + bm - 1) / bm) * ((N + bn - 1) / bn);
        for (int cluster = 1; cluster <= 8; cluster *= 2) {
            // 1, 2, 3, 4, 6, 8, 12, ... slices: a finer search costs the host 17 us per layer and gains nothing
            for (int step = 1; step <= (mode == 2 ? 128 : 1); step = step < 3 ? step + 1 : (step & (step - 1)) ? step / 3 * 4 : step / 2 * 3) {
                const int per = ((K + cluster * step - 1) / (cluster * step) + 31) / 32 * 32;
                if (cluster * step > 1 && per < 64) break;
                int slices = step;
                if (cluster * step > 1 && (int64_t)per * (cluster * step - 1) >= K) {
                    if (vectors || mode != 2) continue;
                    slices = (int)((K + (int64_t)per * cluster - 1) / ((int64_t)per * cluster));      // rounding up leaves fewer
                }
                const int64_t ctas = tiles * cluster * slices;
                const double outputs = (double)M * N;
                const double clk = vectors ? clocks_of_chunks(mode, value_bytes, t, ctas, per, cluster, slices, outputs)
                                           : clocks_of_values(mode, value_bytes, t, bm, bn, ctas, per, cluster, slices, outputs);
                if (clk < best_t) { best_t = clk; best = Plan{t, cluster, slices, per, wide}; }
            }
        }
    }
    return best;
}
}  // namespace simt

constexpr int BN_MAX_BLOCKS = 148 * 8;        // partial rows of batch-norm sums
static bool whole_chunks(int dtype, int channels, const void* p) { return channels % (dtype == CKPT_DTYPE_BF16 ? 8 : 4) == 0 && (uintptr_t)p % 16 == 0; }

// How a call's operands are fetched: each in 16-byte chunks or value by value.  wide: chunks through a filter of more than 16 rows,
// whose mask of places inside the tensor outgrows the 32 bits that the kernel keeps (us, float32, forward / input gradient, value by
// value -> so: 17 x 17 64 -> 64 at 32 x 32, 8 images 937/1255 -> 625/627, 31 x 31 16 -> 32 at 64 x 64, 4 images 1059/2506 -> 558/720).
struct Fetch { bool a, b, wide; };
static Fetch fetch_of(int mode, int dtype, const ConvGeom& g, const void* a, const void* b) {
    Fetch f{whole_chunks(dtype, mode == 0 ? g.cin : g.cout, a), whole_chunks(dtype, g.cin, b), false};
    if (mode == 0) f.a = f.b = f.a && f.b;
    f.wide = mode != 2 && f.a && g.k > 16;
    return f;
}
struct Product { int M, N, K; };
static Product product_of(int mode, const ConvGeom& g) {
    // (a strided layer's K splits over the parity classes of the input: the longest class has ceil(k / stride)^2 positions)
    const int taps = (g.k + g.stride - 1) / g.stride;
    if (mode == 0) return {g.n * g.ho * g.wo, g.cout, g.k * g.k * g.cin};
    if (mode == 1) return {g.n * g.h * g.w, g.cin, taps * taps * g.cout};
    return {g.cout, g.k * g.k * g.cin, g.n * g.ho * g.wo};
}
static simt::Plan plan_of(int mode, int dtype, const ConvGeom& g, const Fetch& f) {
    const Product p = product_of(mode, g);
    return simt::plan(mode, dtype_size(dtype), p.M, p.N, p.K, f.a && f.b, f.wide);
}
static int simt_conv(int mode, int dtype, const ConvGeom& g, const void* a, const void* b, void* out, const float* bias, int relu, const Fetch& f,
                     const simt::Plan& p, cudaStream_t st, const SgdUpdate& upd = SgdUpdate(), float* sums = nullptr) {
    const Product m = product_of(mode, g);
    return dtype == CKPT_DTYPE_BF16 ? simt::launch<__nv_bfloat16>(mode, g, a, b, out, bias, relu, m.M, m.N, m.K, f.a, f.b, p, upd, st, sums)
                                    : simt::launch<float>(mode, g, a, b, out, bias, relu, m.M, m.N, m.K, f.a, f.b, p, upd, st, sums);
}

int simt_conv_fwd(int dtype, const ConvGeom& g, const void* x, const void* w, void* z, const float* bias, int relu, void* stream) {
    if (!bias && !relu && small_conv_supported(dtype, g) && g.cout % 64 == 0) return small_conv_fwd(g, x, w, z, stream);
    const Fetch f = fetch_of(0, dtype, g, x, w);
    return simt_conv(0, dtype, g, x, w, z, bias, relu, f, plan_of(0, dtype, g, f), (cudaStream_t)stream);
}
int simt_conv_fwd_stats(int dtype, const ConvGeom& g, const void* x, const void* w, void* z, float* partial, int* blocks, void* stream) {
    const Fetch f = fetch_of(0, dtype, g, x, w);
    const simt::Plan p = plan_of(0, dtype, g, f);
    const int64_t tile = simt::kShapes[0][p.tile].m, rows = (product_of(0, g).M + tile - 1) / tile * p.cluster;
    *blocks = 0;
    // (the first layer's kernel of its own gathers none; more partial rows than the scratch region is sized for neither)
    if ((small_conv_supported(dtype, g) && g.cout % 64 == 0) || rows > BN_MAX_BLOCKS) return simt_conv_fwd(dtype, g, x, w, z, nullptr, 0, stream);
    *blocks = (int)rows;
    return simt_conv(0, dtype, g, x, w, z, nullptr, 0, f, p, (cudaStream_t)stream, SgdUpdate(), partial);
}
int simt_conv_dgrad(int dtype, const ConvGeom& g, const void* dz, const void* w, void* dx, void* stream) {
    const Fetch f = fetch_of(1, dtype, g, dz, w);
    return simt_conv(1, dtype, g, dz, w, dx, nullptr, 0, f, plan_of(1, dtype, g, f), (cudaStream_t)stream);
}

int simt_selftest_plan(const ConvGeom& g, int dtype, int mode, bool aligned, int32_t* plan) {
    const void* const operand = aligned ? nullptr : (const void*)4;
    const Fetch f = fetch_of(mode, dtype, g, operand, operand);
    const simt::Plan p = plan_of(mode, dtype, g, f);
    const simt::TileShape& s = simt::kShapes[mode][p.tile];
    plan[0] = s.m; plan[1] = s.n; plan[2] = p.cluster; plan[3] = p.slices; plan[4] = p.k_per_slice; plan[5] = s.held[dtype == CKPT_DTYPE_BF16];
    plan[6] = (f.a ? 1 : 0) | (f.b ? 2 : 0) | (f.wide ? 4 : 0);
    return CKPT_OK;
}

int64_t simt_wgrad_scratch_bytes(int dtype, const ConvGeom& g) {
    const Product m = product_of(2, g);
    const int slices = std::max(plan_of(2, dtype, g, {true, true, false}).slices, plan_of(2, dtype, g, {false, false, false}).slices);
    return slices <= 1 ? 0 : (int64_t)slices * m.M * m.N * (int64_t)sizeof(float);
}
int simt_conv_wgrad(int dtype, const ConvGeom& g, const void* dz, const void* x, float* dw, void* scratch, int64_t scratch_bytes, void* stream,
                    const SgdUpdate& upd) {
    const Fetch f = fetch_of(2, dtype, g, dz, x);
    const simt::Plan p = plan_of(2, dtype, g, f);
    const Product m = product_of(2, g);
    const int64_t elems = (int64_t)m.M * m.N;
    if (p.slices > 1 && (!scratch || scratch_bytes < p.slices * elems * 4)) { set_error("wgrad scratch too small"); return CKPT_E_WORKSPACE; }
    int rc = simt_conv(2, dtype, g, dz, x, p.slices > 1 ? scratch : dw, nullptr, 0, f, p, (cudaStream_t)stream, p.slices > 1 ? SgdUpdate() : upd);
    if (rc || p.slices <= 1) return rc;
    return slice_sum((const float*)scratch, dw, elems, p.slices, stream, upd);
}

// ================================================================================================
// Batch normalisation (training mode) + ReLU over a [rows][c] matrix, c contiguous.
// Each thread owns VEC consecutive channels (one 16-byte load when the channel count allows it) and
// walks down the rows of its block's slab; partial sums are combined in a fixed order.
// ================================================================================================
static unsigned elementwise_grid(int64_t items) {
    int64_t b = (items + 255) / 256;
    return (unsigned)std::max<int64_t>(1, std::min<int64_t>(b, 148 * 16));
}

constexpr int BN_THREADS = 256;
constexpr int POOL_BN_BLOCKS = 148 * 2;      // what the device holds of the pooling's sums at once; each leaves two partial rows
static_assert(2 * POOL_BN_BLOCKS <= BN_MAX_BLOCKS, "partial rows of the pooling's sums");
constexpr float BN_EPS = 1e-5f;

// Launch shape of the streaming element-wise kernels: a block works through `per_block` consecutive
// chunks of THREADS*U vectors.  Few chunks per block on large tensors (many short-lived blocks keep
// the memory system busier than a grid that marches in lock step), one per block on small ones.
struct StreamGrid { unsigned blocks; int per_block; };
static StreamGrid stream_grid(int64_t vecs, int threads, int unroll) {
    const int64_t chunk = (int64_t)threads * unroll;
    const int64_t chunks = std::max<int64_t>(1, (vecs + chunk - 1) / chunk);
    StreamGrid g;
    g.per_block = (int)std::max<int64_t>(1, std::min<int64_t>(4, chunks / (148 * 8)));
    g.blocks = (unsigned)((chunks + g.per_block - 1) / g.per_block);
    return g;
}

struct BnLayout {
    int lanes;          // threads across the channel dimension (c / VEC)
    int rows_per_iter;  // rows covered by one sweep of a block
    int blocks;         // row slabs
    int64_t rows_per_block;
};
static BnLayout bn_layout(int64_t rows, int c, int vec) {
    BnLayout L;
    L.lanes = c / vec;
    int lanes_in_block = std::min(L.lanes, BN_THREADS);
    L.rows_per_iter = std::max(1, BN_THREADS / lanes_in_block);
    int64_t want = (rows + (int64_t)L.rows_per_iter * 8 - 1) / ((int64_t)L.rows_per_iter * 8);   // >= 8 sweeps each
    L.blocks = (int)std::max<int64_t>(1, std::min<int64_t>(BN_MAX_BLOCKS, want));
    L.rows_per_block = (rows + L.blocks - 1) / L.blocks;
    L.blocks = (int)((rows + L.rows_per_block - 1) / L.rows_per_block);
    return L;
}
static int bn_vec(int dtype, int c) {
    if (dtype == CKPT_DTYPE_BF16) return (c % 8 == 0) ? 8 : 1;
    return (c % 4 == 0) ? 4 : 1;
}
int64_t bn_scratch_bytes(int64_t rows, int c) {
    (void)rows;
    return (int64_t)BN_MAX_BLOCKS * c * 2 * (int64_t)sizeof(float) + 4 * (int64_t)c * sizeof(float);
}

// Two running sums per channel over a slab of rows.  WHAT 0: (z, z^2).  WHAT 1: (g, g*z) with
// g = dy masked by the ReLU of the forward output (the normalised form g*xhat follows in the
// finalize step: sum g*xhat = inv_std * (sum g*z - mean * sum g)).
template <typename T, int VEC, int WHAT>
__global__ void __launch_bounds__(BN_THREADS, 3) bn_partial_kernel(const T* z, const T* dy,
                                                                   const float* stats, int relu, int64_t rows,
                                                                   int c, int lanes, int rows_per_iter, int64_t rows_per_block,
                                                                   float* partial) {
    previous_grid_done();
    next_grid_may_start();
    extern __shared__ float red[];          // [BN_THREADS][2*VEC]
    constexpr int U = WHAT == 0 ? 4 : 2;    // rows in flight per thread
    const int lanes_here = min(lanes, BN_THREADS);
    const int64_t row_begin = (int64_t)blockIdx.x * rows_per_block;
    const int64_t row_end = min(rows, row_begin + rows_per_block);
    for (int lane0 = 0; lane0 < lanes; lane0 += lanes_here) {
        const int lane = lane0 + threadIdx.x % lanes_here;
        const int r = threadIdx.x / lanes_here;
        float s0[VEC], s1[VEC];
#pragma unroll
        for (int i = 0; i < VEC; ++i) { s0[i] = 0.f; s1[i] = 0.f; }
        const bool active = r < rows_per_iter && lane < lanes;
        if (active) {
            const int ch = lane * VEC;
            float sc[VEC], sh[VEC];
            if (WHAT == 1) {
#pragma unroll
                for (int i = 0; i < VEC; ++i) { sc[i] = stats[2 * c + ch + i]; sh[i] = stats[3 * c + ch + i]; }
            }
            // U rows in flight per thread; sums are still taken in row order
            for (int64_t row = row_begin + r; row < row_end; row += U * (int64_t)rows_per_iter) {
                float v[U][VEC], g[WHAT == 1 ? U : 1][VEC];
#pragma unroll
                for (int u = 0; u < U; ++u) {
                    const int64_t rr = row + (int64_t)u * rows_per_iter;
                    if (rr < row_end) {
                        load_vec<T, VEC>(z + rr * c + ch, v[u]);
                        if (WHAT == 1) load_vec<T, VEC>(dy + rr * c + ch, g[WHAT == 1 ? u : 0]);
                    }
                }
#pragma unroll
                for (int u = 0; u < U; ++u) {
                    if (row + (int64_t)u * rows_per_iter >= row_end) break;
                    if (WHAT == 0) {
#pragma unroll
                        for (int i = 0; i < VEC; ++i) { s0[i] += v[u][i]; s1[i] = fmaf(v[u][i], v[u][i], s1[i]); }
                    } else {
#pragma unroll
                        for (int i = 0; i < VEC; ++i) {
                            float yv = fmaf(v[u][i], sc[i], sh[i]);
                            bool pass = !relu || (float)cvt<T>(fmaxf(yv, 0.f)) > 0.f;
                            float gi = pass ? g[WHAT == 1 ? u : 0][i] : 0.f;
                            s0[i] += gi;
                            s1[i] = fmaf(gi, v[u][i], s1[i]);
                        }
                    }
                }
            }
        }
        float* mine = red + ((size_t)(threadIdx.x / lanes_here) * lanes_here + threadIdx.x % lanes_here) * 2 * VEC;
#pragma unroll
        for (int i = 0; i < VEC; ++i) { mine[i] = s0[i]; mine[VEC + i] = s1[i]; }
        __syncthreads();
        if (r == 0 && lane < lanes) {
            const int ch = lane * VEC;
#pragma unroll
            for (int i = 0; i < VEC; ++i) {
                float a = 0.f, b = 0.f;
                for (int rr = 0; rr < rows_per_iter; ++rr) {
                    const float* o = red + ((size_t)rr * lanes_here + threadIdx.x % lanes_here) * 2 * VEC;
                    a += o[i];
                    b += o[VEC + i];
                }
                partial[((size_t)blockIdx.x * 2 + 0) * c + ch + i] = a;
                partial[((size_t)blockIdx.x * 2 + 1) * c + ch + i] = b;
            }
        }
        __syncthreads();
    }
}

// Sums of the per-block partials of 8 channels (32 bytes of a row) by one block: 64 threads share a channel, ten row pairs
// each in flight at once, every sum as two floats (twice float precision), combined in a fixed order.  Latency is all there
// is to it, the arithmetic behind the loads included: steps past the last row are left out, and 32 lanes share the adding up
// of the warps' sums (batch norm forward of 25088 x 64, us: one channel per warp in doubles 8.8, eight lanes adding up sixteen
// warps in turn 9.6, this 9.2; backward by separate kernels 13.0 -> 12.3).
constexpr int FIN_CH = 8, FIN_ROWS = 64, FIN_THREADS = FIN_CH * FIN_ROWS;
__device__ __forceinline__ bool block_channel_sums(const float* partial, int blocks, int c, int ch, double& s, double& q) {
    __shared__ float4 red[FIN_THREADS / 32][FIN_CH];
    const int row = threadIdx.x / FIN_CH, warp = threadIdx.x / 32, lane = threadIdx.x % 32;
    float2 a = make_float2(0.f, 0.f), b = make_float2(0.f, 0.f);
    constexpr int U = 10;
    for (int r0 = 0; r0 < blocks; r0 += U * FIN_ROWS) {
        float x[U], y[U];
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const int r = r0 + u * FIN_ROWS + row;
            const bool in = r < blocks && ch < c;
            x[u] = in ? partial[(size_t)r * 2 * c + ch] : 0.f;
            y[u] = in ? partial[((size_t)r * 2 + 1) * c + ch] : 0.f;
        }
#pragma unroll
        for (int u = 0; u < U; ++u) {
            if (r0 + u * FIN_ROWS >= blocks) break;
            two_sum(a, x[u]); two_sum(b, y[u]);
        }
    }
    auto over_lanes = [&]() {                                  // lanes with the same channel
#pragma unroll
        for (int o = 16; o >= FIN_CH; o >>= 1) {
            const float ax = __shfl_xor_sync(0xffffffffu, a.x, o), ay = __shfl_xor_sync(0xffffffffu, a.y, o);
            const float bx = __shfl_xor_sync(0xffffffffu, b.x, o), by = __shfl_xor_sync(0xffffffffu, b.y, o);
            two_sum(a, ax); a.y += ay;
            two_sum(b, bx); b.y += by;
        }
    };
    over_lanes();
    if (lane < FIN_CH) red[warp][lane] = make_float4(a.x, a.y, b.x, b.y);
    __syncthreads();
    if (warp != 0) return false;
    a = b = make_float2(0.f, 0.f);
#pragma unroll
    for (int w = 0; w < FIN_THREADS / 32; w += 4) {
        const float4 o = red[w + lane / FIN_CH][lane % FIN_CH];
        two_sum(a, o.x); a.y += o.y;
        two_sum(b, o.z); b.y += o.w;
    }
    over_lanes();
    if (lane >= FIN_CH || ch >= c) return false;
    s = (double)a.x + a.y; q = (double)b.x + b.y;
    return true;
}

// mean, 1/sqrt(var+eps), scale = gamma*inv, shift = beta - mean*scale.
__global__ void __launch_bounds__(FIN_THREADS) bn_finalize_fwd_kernel(const float* partial, int blocks, int c, double inv_rows,
                                       const float* gamma, const float* beta, float* stats) {
    previous_grid_done();
    next_grid_may_start();
    const int ch = blockIdx.x * FIN_CH + threadIdx.x % FIN_CH;
    const float g = ch < c ? gamma[ch] : 0.f, b = ch < c ? beta[ch] : 0.f;
    double s, q;
    if (!block_channel_sums(partial, blocks, c, ch, s, q)) return;
    double mean = s * inv_rows;
    double var = q * inv_rows - mean * mean;
    if (var < 0.0) var = 0.0;
    float inv = (float)(1.0 / sqrt(var + (double)BN_EPS));
    float scale = g * inv;
    stats[ch] = (float)mean;
    stats[c + ch] = inv;
    stats[2 * c + ch] = scale;
    stats[3 * c + ch] = b - (float)mean * scale;
}

// dbeta, dgamma and the two per-channel coefficients of the input gradient:
//   dz = scale*g - k1 - xhat*k2,  k1 = scale*dbeta/rows, k2 = scale*dgamma/rows
__global__ void __launch_bounds__(FIN_THREADS) bn_finalize_bwd_kernel(const float* partial, int blocks, int c, double inv_rows,
                                       const float* stats, float* dgamma, float* dbeta,
                                       float* coef, SgdUpdate gamma, SgdUpdate beta) {
    previous_grid_done();
    next_grid_may_start();
    const int ch = blockIdx.x * FIN_CH + threadIdx.x % FIN_CH;
    double s, q;
    if (!block_channel_sums(partial, blocks, c, ch, s, q)) return;
    // q = sum g*z  ->  sum g*xhat = inv_std * (q - mean * sum g)
    const double gx = (double)stats[c + ch] * (q - (double)stats[ch] * s);
    dbeta[ch] = (float)s;
    dgamma[ch] = (float)gx;
    if (gamma.w) { float* w = (float*)gamma.w + ch; *w = fmaf(-gamma.lr, (float)gx, *w); }
    if (beta.w) { float* w = (float*)beta.w + ch; *w = fmaf(-beta.lr, (float)s, *w); }
    double scale = stats[2 * c + ch];
    // dz = scale*g - k1 - xhat*k2 with k1 = scale*dbeta/rows, k2 = scale*dgamma/rows and
    // xhat = (z - mean)*inv_std, regrouped as  dz = scale*g - A - z*B
    const double k1 = scale * s * inv_rows, k2 = scale * gx * inv_rows;
    const double mean = stats[ch], inv = stats[c + ch];
    coef[ch] = (float)(k1 - mean * inv * k2);
    coef[c + ch] = (float)(inv * k2);
}

// y = max(z*scale + shift, 0).  A block walks consecutive chunks of 256*U vectors; when the block size
// is a multiple of the number of channel groups every thread stays on one channel group, keeps its
// coefficients in registers and has U packed 16-byte loads in flight.
constexpr int BN_APPLY_U = 8;
template <typename T, int VEC>
__global__ void __launch_bounds__(256, 4) bn_apply_kernel(const T* z, const float* stats, int relu,
                                                          int64_t vecs, int lanes, int c, int per_block, T* y) {
    previous_grid_done();
    next_grid_may_start();
    constexpr int U = BN_APPLY_U;
    const int64_t chunk = 256 * U;
    const int64_t begin = (int64_t)blockIdx.x * per_block * chunk;
    if (256 % lanes == 0) {
        const int ch = (int)(threadIdx.x % lanes) * VEC;
        float sc[VEC], sh[VEC];
#pragma unroll
        for (int k = 0; k < VEC; ++k) { sc[k] = stats[2 * c + ch + k]; sh[k] = stats[3 * c + ch + k]; }
        for (int it = 0; it < per_block; ++it) {
            const int64_t i0 = begin + it * chunk + threadIdx.x;
            if (i0 >= vecs) break;
            RawVec<T, VEC> r[U];
#pragma unroll
            for (int u = 0; u < U; ++u)
                if (i0 + u * 256 < vecs) r[u] = load_raw<T, VEC>(z + (i0 + u * 256) * VEC);
#pragma unroll
            for (int u = 0; u < U; ++u) {
                if (i0 + u * 256 >= vecs) break;
                float v[VEC], o[VEC];
                unpack<T, VEC>(r[u], v);
#pragma unroll
                for (int k = 0; k < VEC; ++k) {
                    float t = fmaf(v[k], sc[k], sh[k]);
                    o[k] = relu ? fmaxf(t, 0.f) : t;
                }
                store_vec<T, VEC>(y + (i0 + u * 256) * VEC, o);
            }
        }
        return;
    }
    const int64_t end = min(vecs, begin + per_block * chunk);
    for (int64_t i = begin + threadIdx.x; i < end; i += 256) {
        const int ch = (int)(i % lanes) * VEC;
        float v[VEC], o[VEC];
        load_vec<T, VEC>(z + i * VEC, v);
#pragma unroll
        for (int k = 0; k < VEC; ++k) {
            float t = fmaf(v[k], stats[2 * c + ch + k], stats[3 * c + ch + k]);
            o[k] = relu ? fmaxf(t, 0.f) : t;
        }
        store_vec<T, VEC>(y + i * VEC, o);
    }
}

template <typename T, int VEC>
__device__ __forceinline__ void bn_bwd_point(const float (&v)[VEC], const float (&g)[VEC], const float (&sc)[VEC],
                                             const float (&sh)[VEC], const float (&ca)[VEC], const float (&cb)[VEC], int relu,
                                             float (&o)[VEC]) {
#pragma unroll
    for (int k = 0; k < VEC; ++k) {
        float yv = fmaf(v[k], sc[k], sh[k]);
        bool pass = !relu || (float)cvt<T>(fmaxf(yv, 0.f)) > 0.f;
        float gi = pass ? g[k] : 0.f;
        o[k] = fmaf(-v[k], cb[k], fmaf(sc[k], gi, -ca[k]));
    }
}

constexpr int BN_BWD_U = 4;
template <typename T, int VEC>
__global__ void __launch_bounds__(256, 3) bn_bwd_apply_kernel(const T* dy, const T* z,
                                                              const float* stats, const float* coef,
                                                              int relu, int64_t vecs, int lanes, int c, int per_block,
                                                              T* dz) {
    previous_grid_done();
    next_grid_may_start();
    constexpr int U = BN_BWD_U;
    const int64_t chunk = 256 * U;
    const int64_t begin = (int64_t)blockIdx.x * per_block * chunk;
    float sc[VEC], sh[VEC], ca[VEC], cb[VEC];
    auto load_coef = [&](int ch) {
#pragma unroll
        for (int k = 0; k < VEC; ++k) {
            sc[k] = stats[2 * c + ch + k]; sh[k] = stats[3 * c + ch + k];
            ca[k] = coef[ch + k]; cb[k] = coef[c + ch + k];
        }
    };
    if (256 % lanes == 0) {
        load_coef((int)(threadIdx.x % lanes) * VEC);
        for (int it = 0; it < per_block; ++it) {
            const int64_t i0 = begin + it * chunk + threadIdx.x;
            if (i0 >= vecs) break;
            RawVec<T, VEC> rv[U], rg[U];
#pragma unroll
            for (int u = 0; u < U; ++u)
                if (i0 + u * 256 < vecs) { rv[u] = load_raw<T, VEC>(z + (i0 + u * 256) * VEC); rg[u] = load_raw<T, VEC>(dy + (i0 + u * 256) * VEC); }
#pragma unroll
            for (int u = 0; u < U; ++u) {
                if (i0 + u * 256 >= vecs) break;
                float v[VEC], g[VEC], o[VEC];
                unpack<T, VEC>(rv[u], v);
                unpack<T, VEC>(rg[u], g);
                bn_bwd_point<T, VEC>(v, g, sc, sh, ca, cb, relu, o);
                store_vec<T, VEC>(dz + (i0 + u * 256) * VEC, o);
            }
        }
        return;
    }
    const int64_t end = min(vecs, begin + per_block * chunk);
    for (int64_t i = begin + threadIdx.x; i < end; i += 256) {
        load_coef((int)(i % lanes) * VEC);
        float v[VEC], g[VEC], o[VEC];
        load_vec<T, VEC>(z + i * VEC, v);
        load_vec<T, VEC>(dy + i * VEC, g);
        bn_bwd_point<T, VEC>(v, g, sc, sh, ca, cb, relu, o);
        store_vec<T, VEC>(dz + i * VEC, o);
    }
}

// Streaming form of the per-channel sums for channel counts whose vector lanes divide the block:
// every thread keeps one channel group for the whole kernel (its stride through the tensor is a
// multiple of the row length), holds U independent 16-byte loads in flight, and the block combines
// its threads by a fixed tree.  Same two sums as bn_partial_kernel.
constexpr int BNF_THREADS = 384;
template <typename T, int VEC, int WHAT>
__global__ void __launch_bounds__(BNF_THREADS, 2) bn_partial_stream_kernel(const T* z, const T* dy,
                                                                           const float* stats, int relu,
                                                                           int64_t vecs, int lanes, int c,
                                                                           float* partial) {
    previous_grid_done();
    next_grid_may_start();
    __shared__ float red[BNF_THREADS][2 * VEC + 1];
    constexpr int U = WHAT == 0 ? 8 : 4;
    const int64_t stride = (int64_t)gridDim.x * BNF_THREADS;
    const int64_t first = (int64_t)blockIdx.x * BNF_THREADS + threadIdx.x;
    const int ch = (int)(first % lanes) * VEC;
    float s0[VEC], s1[VEC], sc[VEC], sh[VEC];
#pragma unroll
    for (int k = 0; k < VEC; ++k) { s0[k] = 0.f; s1[k] = 0.f; }
    if (WHAT == 1) {
#pragma unroll
        for (int k = 0; k < VEC; ++k) { sc[k] = stats[2 * c + ch + k]; sh[k] = stats[3 * c + ch + k]; }
    }
    for (int64_t i = first; i < vecs; i += U * stride) {
        RawVec<T, VEC> rv[U], rg[WHAT == 1 ? U : 1];
#pragma unroll
        for (int u = 0; u < U; ++u) {
            if (i + u * stride < vecs) {
                rv[u] = load_raw<T, VEC>(z + (i + u * stride) * VEC);
                if (WHAT == 1) rg[WHAT == 1 ? u : 0] = load_raw<T, VEC>(dy + (i + u * stride) * VEC);
            }
        }
#pragma unroll
        for (int u = 0; u < U; ++u) {
            if (i + u * stride >= vecs) break;
            float v[VEC], g[VEC];
            unpack<T, VEC>(rv[u], v);
            if (WHAT == 1) unpack<T, VEC>(rg[WHAT == 1 ? u : 0], g);
#pragma unroll
            for (int k = 0; k < VEC; ++k) {
                if (WHAT == 0) {
                    s0[k] += v[k];
                    s1[k] = fmaf(v[k], v[k], s1[k]);
                } else {
                    float yv = fmaf(v[k], sc[k], sh[k]);
                    bool pass = !relu || (float)cvt<T>(fmaxf(yv, 0.f)) > 0.f;
                    float gi = pass ? g[k] : 0.f;
                    s0[k] += gi;
                    s1[k] = fmaf(gi, v[k], s1[k]);
                }
            }
        }
    }
#pragma unroll
    for (int k = 0; k < VEC; ++k) { red[threadIdx.x][k] = s0[k]; red[threadIdx.x][VEC + k] = s1[k]; }
    __syncthreads();
    // 384 -> 128 partial rows, then halving down to one row per channel group; threads t and t + m*lanes
    // always hold the same channel group because every step keeps the index modulo `lanes`
    if (threadIdx.x < 128) {
#pragma unroll
        for (int k = 0; k < 2 * VEC; ++k) red[threadIdx.x][k] = (red[threadIdx.x][k] + red[threadIdx.x + 128][k]) + red[threadIdx.x + 256][k];
    }
    __syncthreads();
    for (int off = 64; off >= lanes; off >>= 1) {
        if ((int)threadIdx.x < off) {
#pragma unroll
            for (int k = 0; k < 2 * VEC; ++k) red[threadIdx.x][k] += red[threadIdx.x + off][k];
        }
        __syncthreads();
    }
    if ((int)threadIdx.x < lanes) {
        const int chn = (int)(((int64_t)blockIdx.x * BNF_THREADS + threadIdx.x) % lanes) * VEC;
#pragma unroll
        for (int k = 0; k < VEC; ++k) {
            partial[((size_t)blockIdx.x * 2 + 0) * c + chn + k] = red[threadIdx.x][k];
            partial[((size_t)blockIdx.x * 2 + 1) * c + chn + k] = red[threadIdx.x][VEC + k];
        }
    }
}

// The streaming kernel needs: lanes a power of two between 8 and 128 (so that 128 and the block
// size are multiples of it).
static bool bn_stream_ok(int lanes) { return lanes >= 8 && lanes <= 128 && (lanes & (lanes - 1)) == 0; }
static int bn_stream_blocks(int64_t vecs) {
    int64_t b = (vecs + (int64_t)BNF_THREADS * 8 - 1) / ((int64_t)BNF_THREADS * 8);
    return (int)std::max<int64_t>(1, std::min<int64_t>(b, 148 * 2));
}

template <typename T, int VEC>
static int bn_stats_t(int64_t rows, int c, const void* z, const float* gamma, const float* beta, float* stats, void* scratch,
                      cudaStream_t st) {
    BnLayout L = bn_layout(rows, c, VEC);
    float* partial = (float*)scratch;
    int blocks = L.blocks;
    if (VEC > 1 && bn_stream_ok(L.lanes)) {
        const int64_t vecs = rows * c / VEC;
        blocks = bn_stream_blocks(vecs);
        launch(Start::ON_STREAMS, bn_partial_stream_kernel<T, VEC, 0>, blocks, BNF_THREADS, 0, st, (const T*)z, nullptr, nullptr, 0, vecs, L.lanes, c, partial);
    } else {
        size_t smem = (size_t)BN_THREADS * 2 * VEC * sizeof(float);
        launch(Start::ON_STREAMS, bn_partial_kernel<T, VEC, 0>, L.blocks, BN_THREADS, smem, st, (const T*)z, nullptr, nullptr, 0, rows, c, L.lanes,
                                                                          L.rows_per_iter, L.rows_per_block, partial);
    }
    CKPT_LAUNCH_CHECK("batch-norm statistics");
    launch(Start::ON_STREAMS, bn_finalize_fwd_kernel, (c + FIN_CH - 1) / FIN_CH, FIN_THREADS, 0, st, partial, blocks, c, 1.0 / (double)rows, gamma, beta, stats);
    CKPT_LAUNCH_CHECK("batch-norm finalize");
    return CKPT_OK;
}

template <typename T, int VEC>
static int bn_apply_t(int64_t rows, int c, const void* z, const float* stats, int relu, void* y, cudaStream_t st) {
    int64_t vecs = rows * c / VEC;
    const StreamGrid sg = stream_grid(vecs, 256, BN_APPLY_U);
    launch(Start::ON_STREAMS, bn_apply_kernel<T, VEC>, sg.blocks, 256, 0, st, (const T*)z, stats, relu, vecs, c / VEC, c, sg.per_block, (T*)y);
    CKPT_LAUNCH_CHECK("batch-norm apply");
    return CKPT_OK;
}

template <typename T, int VEC>
static int bn_backward_t(int64_t rows, int c, const void* dy, const void* z, const float* stats, int relu, void* dz,
                         float* dgamma, float* dbeta, void* scratch, const BnBackwardExtra& ex, cudaStream_t st) {
    BnLayout L = bn_layout(rows, c, VEC);
    float* partial = (float*)scratch;
    float* coef = partial + (size_t)BN_MAX_BLOCKS * c * 2;
    int blocks = L.blocks;
    if (VEC > 1 && bn_stream_ok(L.lanes)) {
        const int64_t nvecs = rows * c / VEC;
        blocks = bn_stream_blocks(nvecs);
        launch(Start::ON_STREAMS, bn_partial_stream_kernel<T, VEC, 1>, blocks, BNF_THREADS, 0, st, (const T*)z, (const T*)dy, stats, relu, nvecs, L.lanes, c, partial);
    } else {
        size_t smem = (size_t)BN_THREADS * 2 * VEC * sizeof(float);
        launch(Start::ON_STREAMS, bn_partial_kernel<T, VEC, 1>, L.blocks, BN_THREADS, smem, st, (const T*)z, (const T*)dy, stats, relu, rows, c, L.lanes,
                                                                          L.rows_per_iter, L.rows_per_block, partial);
    }
    CKPT_LAUNCH_CHECK("batch-norm backward sums");
    launch(Start::ON_STREAMS, bn_finalize_bwd_kernel, (c + FIN_CH - 1) / FIN_CH, FIN_THREADS, 0, st, partial, blocks, c, 1.0 / (double)rows, stats, dgamma, dbeta, coef, ex.gamma, ex.beta);
    CKPT_LAUNCH_CHECK("batch-norm backward finalize");
    int64_t vecs = rows * c / VEC;
    const StreamGrid sg = stream_grid(vecs, 256, BN_BWD_U);
    launch(Start::ON_STREAMS, bn_bwd_apply_kernel<T, VEC>, sg.blocks, 256, 0, st, (const T*)dy, (const T*)z, stats, coef, relu, vecs, L.lanes, c,
                                                           sg.per_block, (T*)dz);
    CKPT_LAUNCH_CHECK("batch-norm backward apply");
    return CKPT_OK;
}

// Statistics from partial sums that another kernel (a convolution epilogue) has already written:
// partial = [blocks][sum | sum of squares][c] floats.
int bn_statistics_from_partials(const float* partial, int blocks, int64_t rows, int c, const float* gamma, const float* beta,
                                float* stats, void* stream) {
    launch(Start::ON_STREAMS, bn_finalize_fwd_kernel, (c + FIN_CH - 1) / FIN_CH, FIN_THREADS, 0, (cudaStream_t)stream, partial, blocks, c, 1.0 / (double)rows, gamma, beta, stats);
    CKPT_LAUNCH_CHECK("batch-norm finalize");
    return CKPT_OK;
}

int bn_statistics(int dtype, int64_t rows, int c, const void* z, const float* gamma, const float* beta, float* stats,
                  void* scratch, void* stream) {
    cudaStream_t st = (cudaStream_t)stream;
    int vec = bn_vec(dtype, c);
    if (dtype == CKPT_DTYPE_BF16)
        return vec == 8 ? bn_stats_t<__nv_bfloat16, 8>(rows, c, z, gamma, beta, stats, scratch, st)
                        : bn_stats_t<__nv_bfloat16, 1>(rows, c, z, gamma, beta, stats, scratch, st);
    return vec == 4 ? bn_stats_t<float, 4>(rows, c, z, gamma, beta, stats, scratch, st)
                    : bn_stats_t<float, 1>(rows, c, z, gamma, beta, stats, scratch, st);
}

int bn_apply(int dtype, int64_t rows, int c, const void* z, const float* stats, int relu, void* y, void* stream) {
    cudaStream_t st = (cudaStream_t)stream;
    int vec = bn_vec(dtype, c);
    if (dtype == CKPT_DTYPE_BF16)
        return vec == 8 ? bn_apply_t<__nv_bfloat16, 8>(rows, c, z, stats, relu, y, st) : bn_apply_t<__nv_bfloat16, 1>(rows, c, z, stats, relu, y, st);
    return vec == 4 ? bn_apply_t<float, 4>(rows, c, z, stats, relu, y, st) : bn_apply_t<float, 1>(rows, c, z, stats, relu, y, st);
}

int bn_relu_forward(int dtype, int64_t rows, int c, const void* z, const float* gamma, const float* beta, int relu, void* y,
                    float* stats, void* scratch, void* stream) {
    int rc = bn_statistics(dtype, rows, c, z, gamma, beta, stats, scratch, stream);
    if (rc) return rc;
    return bn_apply(dtype, rows, c, z, stats, relu, y, stream);
}

// Residual join of a bottleneck block: y = max(z*scale + shift + shortcut, 0), where the shortcut is
// either an already activated tensor (stats_sc == nullptr) or a second pre-normalisation tensor with
// its own scale/shift (projection branch).
template <typename T>
__global__ void __launch_bounds__(256) bn_add_relu_kernel(const T* z, const float* stats,
                                                          const T* sc, const float* stats_sc,
                                                          int64_t elems, int c, T* y) {
    previous_grid_done();
    next_grid_may_start();
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < elems; i += (int64_t)gridDim.x * blockDim.x) {
        const int ch = (int)(i % c);
        float v = fmaf(ld(z + i), stats[2 * c + ch], stats[3 * c + ch]);
        float s = ld(sc + i);
        if (stats_sc) s = fmaf(s, stats_sc[2 * c + ch], stats_sc[3 * c + ch]);
        y[i] = cvt<T>(fmaxf(v + s, 0.f));
    }
}
// Vector form: a block walks consecutive chunks of 256*U vectors, every thread stays on one channel group
// (the block size is a multiple of the number of groups) and keeps its coefficients in registers.
constexpr int BN_JOIN_U = 4;
template <typename T, int VEC>
__global__ void __launch_bounds__(256, 3) bn_add_relu_vec_kernel(const T* z, const float* stats,
                                                                 const T* sc, const float* stats_sc,
                                                                 int64_t vecs, int lanes, int c, int per_block, T* y) {
    previous_grid_done();
    next_grid_may_start();
    constexpr int U = BN_JOIN_U;
    const int64_t chunk = 256 * U;
    const int64_t begin = (int64_t)blockIdx.x * per_block * chunk;
    const int ch = (int)(threadIdx.x % lanes) * VEC;
    float a[VEC], b[VEC], as[VEC], bs[VEC];
#pragma unroll
    for (int k = 0; k < VEC; ++k) {
        a[k] = stats[2 * c + ch + k]; b[k] = stats[3 * c + ch + k];
        as[k] = stats_sc ? stats_sc[2 * c + ch + k] : 1.f;
        bs[k] = stats_sc ? stats_sc[3 * c + ch + k] : 0.f;
    }
    for (int it = 0; it < per_block; ++it) {
        const int64_t i0 = begin + it * chunk + threadIdx.x;
        if (i0 >= vecs) break;
        RawVec<T, VEC> rz[U], rs[U];
#pragma unroll
        for (int u = 0; u < U; ++u)
            if (i0 + u * 256 < vecs) { rz[u] = load_raw<T, VEC>(z + (i0 + u * 256) * VEC); rs[u] = load_raw<T, VEC>(sc + (i0 + u * 256) * VEC); }
#pragma unroll
        for (int u = 0; u < U; ++u) {
            if (i0 + u * 256 >= vecs) break;
            float v[VEC], sv[VEC], o[VEC];
            unpack<T, VEC>(rz[u], v);
            unpack<T, VEC>(rs[u], sv);
#pragma unroll
            for (int k = 0; k < VEC; ++k) {
                const float t = fmaf(v[k], a[k], b[k]);
                const float s2 = stats_sc ? fmaf(sv[k], as[k], bs[k]) : sv[k];
                o[k] = fmaxf(t + s2, 0.f);
            }
            store_vec<T, VEC>(y + (i0 + u * 256) * VEC, o);
        }
    }
}
template <typename T, int VEC>
static bool bn_add_relu_vec(int64_t rows, int c, const void* z, const float* stats, const void* shortcut,
                            const float* stats_shortcut, void* y, cudaStream_t st) {
    if (c % VEC || 256 % (c / VEC)) return false;
    const int64_t vecs = rows * c / VEC;
    const StreamGrid sg = stream_grid(vecs, 256, BN_JOIN_U);
    launch(Start::ON_STREAMS, bn_add_relu_vec_kernel<T, VEC>, sg.blocks, 256, 0, st, (const T*)z, stats, (const T*)shortcut, stats_shortcut, vecs, c / VEC, c,
                                                              sg.per_block, (T*)y);
    return true;
}
int bn_add_relu(int dtype, int64_t rows, int c, const void* z, const float* stats, const void* shortcut,
                const float* stats_shortcut, void* y, void* stream) {
    const int64_t elems = rows * c;
    cudaStream_t st = (cudaStream_t)stream;
    if (dtype == CKPT_DTYPE_BF16) {
        if (!bn_add_relu_vec<__nv_bfloat16, 8>(rows, c, z, stats, shortcut, stats_shortcut, y, st))
            launch(Start::ON_STREAMS, bn_add_relu_kernel<__nv_bfloat16>, elementwise_grid(elems), 256, 0, st, 
                (const __nv_bfloat16*)z, stats, (const __nv_bfloat16*)shortcut, stats_shortcut, elems, c, (__nv_bfloat16*)y);
    } else if (!bn_add_relu_vec<float, 4>(rows, c, z, stats, shortcut, stats_shortcut, y, st)) {
        launch(Start::ON_STREAMS, bn_add_relu_kernel<float>, elementwise_grid(elems), 256, 0, st, 
            (const float*)z, stats, (const float*)shortcut, stats_shortcut, elems, c, (float*)y);
    }
    CKPT_LAUNCH_CHECK("residual join");
    return CKPT_OK;
}

template <typename T>
__global__ void __launch_bounds__(256) add_kernel(const T* a, const T* b, T* out, int64_t elems) {
    previous_grid_done();
    next_grid_may_start();
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < elems; i += (int64_t)gridDim.x * blockDim.x)
        out[i] = cvt<T>(ld(a + i) + ld(b + i));
}
// 16-byte form of the sum (out may alias an input); four packed loads per operand in flight.
template <typename T, int VEC>
__global__ void __launch_bounds__(256) add_vec_kernel(const T* a, const T* b, T* out, int64_t vecs) {
    previous_grid_done();
    next_grid_may_start();
    constexpr int U = 4;
    for (int64_t i0 = (int64_t)blockIdx.x * (256 * U) + threadIdx.x; i0 < vecs; i0 += (int64_t)gridDim.x * (256 * U)) {
        RawVec<T, VEC> ra[U], rb[U];
#pragma unroll
        for (int u = 0; u < U; ++u)
            if (i0 + u * 256 < vecs) { ra[u] = load_raw<T, VEC>(a + (i0 + u * 256) * VEC); rb[u] = load_raw<T, VEC>(b + (i0 + u * 256) * VEC); }
#pragma unroll
        for (int u = 0; u < U; ++u) {
            if (i0 + u * 256 >= vecs) break;
            float x[VEC], y[VEC], o[VEC];
            unpack<T, VEC>(ra[u], x);
            unpack<T, VEC>(rb[u], y);
#pragma unroll
            for (int k = 0; k < VEC; ++k) o[k] = x[k] + y[k];
            store_vec<T, VEC>(out + (i0 + u * 256) * VEC, o);
        }
    }
}
static bool aligned16(const void* p) { return ((uintptr_t)p & 15u) == 0; }
int add_tensors(int dtype, int64_t elems, const void* a, const void* b, void* out, void* stream) {
    cudaStream_t st = (cudaStream_t)stream;
    const int vec = dtype == CKPT_DTYPE_BF16 ? 8 : 4;
    if (elems % vec == 0 && aligned16(a) && aligned16(b) && aligned16(out)) {
        const int64_t vecs = elems / vec;
        const unsigned grid = (unsigned)std::max<int64_t>(1, std::min<int64_t>((vecs + 1023) / 1024, 148 * 32));
        if (dtype == CKPT_DTYPE_BF16) launch(Start::ON_STREAMS, add_vec_kernel<__nv_bfloat16, 8>, grid, 256, 0, st, (const __nv_bfloat16*)a, (const __nv_bfloat16*)b, (__nv_bfloat16*)out, vecs);
        else launch(Start::ON_STREAMS, add_vec_kernel<float, 4>, grid, 256, 0, st, (const float*)a, (const float*)b, (float*)out, vecs);
    } else if (dtype == CKPT_DTYPE_BF16) {
        launch(Start::ON_STREAMS, add_kernel<__nv_bfloat16>, elementwise_grid(elems), 256, 0, st, (const __nv_bfloat16*)a, (const __nv_bfloat16*)b, (__nv_bfloat16*)out, elems);
    } else {
        launch(Start::ON_STREAMS, add_kernel<float>, elementwise_grid(elems), 256, 0, st, (const float*)a, (const float*)b, (float*)out, elems);
    }
    CKPT_LAUNCH_CHECK("gradient join");
    return CKPT_OK;
}

int bn_relu_backward(int dtype, int64_t rows, int c, void* dy, const void* z, const float* stats, int relu, void* dz, float* dgamma,
                     float* dbeta, void* scratch, void* stream, const BnBackwardExtra& ex) {
    cudaStream_t st = (cudaStream_t)stream;
    if (ex.counters && ex.status && bn_backward_form(dtype, rows, c, dy, z, ex.mask, dz) != BnForm::separate)
        return bn_backward_fused(dtype, rows, c, dy, z, stats, relu, dz, dgamma, dbeta, (float*)scratch, ex, stream);
    if (ex.mask) {
        int rc = relu_mask_inplace(dtype, rows * c, dy, ex.mask, stream);
        if (rc) return rc;
    }
    int vec = bn_vec(dtype, c);
    if (dtype == CKPT_DTYPE_BF16)
        return vec == 8 ? bn_backward_t<__nv_bfloat16, 8>(rows, c, dy, z, stats, relu, dz, dgamma, dbeta, scratch, ex, st)
                        : bn_backward_t<__nv_bfloat16, 1>(rows, c, dy, z, stats, relu, dz, dgamma, dbeta, scratch, ex, st);
    return vec == 4 ? bn_backward_t<float, 4>(rows, c, dy, z, stats, relu, dz, dgamma, dbeta, scratch, ex, st)
                    : bn_backward_t<float, 1>(rows, c, dy, z, stats, relu, dz, dgamma, dbeta, scratch, ex, st);
}

// Batch-norm backward whose per-channel sums (sum g, sum g*z over `blocks` partial row pairs at the start of
// `scratch`) were left by the kernel that produced dy: finalize and apply only.
template <typename T, int VEC>
static int bn_backward_tail_t(int64_t rows, int c, const void* dy, const void* z, const float* stats, int relu, void* dz,
                              float* dgamma, float* dbeta, void* scratch, int blocks, const BnBackwardExtra& ex, cudaStream_t st) {
    float* partial = (float*)scratch;
    float* coef = partial + (size_t)BN_MAX_BLOCKS * c * 2;
    launch(Start::ON_STREAMS, bn_finalize_bwd_kernel, (c + FIN_CH - 1) / FIN_CH, FIN_THREADS, 0, st, partial, blocks, c, 1.0 / (double)rows, stats, dgamma, dbeta, coef, ex.gamma, ex.beta);
    CKPT_LAUNCH_CHECK("batch-norm backward finalize");
    const int64_t vecs = rows * c / VEC;
    const StreamGrid sg = stream_grid(vecs, 256, BN_BWD_U);
    launch(Start::ON_STREAMS, bn_bwd_apply_kernel<T, VEC>, sg.blocks, 256, 0, st, (const T*)dy, (const T*)z, stats, coef, relu, vecs, c / VEC, c,
                                                           sg.per_block, (T*)dz);
    CKPT_LAUNCH_CHECK("batch-norm backward apply");
    return CKPT_OK;
}
int bn_relu_backward_from_partials(int dtype, int64_t rows, int c, const void* dy, const void* z, const float* stats, int relu,
                                   void* dz, float* dgamma, float* dbeta, void* scratch, int blocks, void* stream,
                                   const BnBackwardExtra& ex) {
    cudaStream_t st = (cudaStream_t)stream;
    if (blocks < 1 || blocks > BN_MAX_BLOCKS) { set_error("batch-norm backward: %d partial rows", blocks); return CKPT_E_BAD_ARG; }
    int vec = bn_vec(dtype, c);
    if (dtype == CKPT_DTYPE_BF16)
        return vec == 8 ? bn_backward_tail_t<__nv_bfloat16, 8>(rows, c, dy, z, stats, relu, dz, dgamma, dbeta, scratch, blocks, ex, st)
                        : bn_backward_tail_t<__nv_bfloat16, 1>(rows, c, dy, z, stats, relu, dz, dgamma, dbeta, scratch, blocks, ex, st);
    return vec == 4 ? bn_backward_tail_t<float, 4>(rows, c, dy, z, stats, relu, dz, dgamma, dbeta, scratch, blocks, ex, st)
                    : bn_backward_tail_t<float, 1>(rows, c, dy, z, stats, relu, dz, dgamma, dbeta, scratch, blocks, ex, st);
}

// ================================================================================================
// Pooling
// ================================================================================================
template <typename T>
__global__ void maxpool_fwd_kernel(const T* x, T* y, int n, int h, int w, int c, int ho, int wo,
                                   int k, int stride, int pad) {
    previous_grid_done();
    next_grid_may_start();
    int64_t total = (int64_t)n * ho * wo * c;
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < total; i += (int64_t)gridDim.x * blockDim.x) {
        int ch = (int)(i % c);
        int64_t t = i / c;
        int ow = (int)(t % wo); t /= wo;
        int oh = (int)(t % ho);
        int img = (int)(t / ho);
        float best = -INFINITY;
        for (int r = 0; r < k; ++r) {
            int ih = oh * stride - pad + r;
            if (ih < 0 || ih >= h) continue;
            for (int s = 0; s < k; ++s) {
                int iw = ow * stride - pad + s;
                if (iw < 0 || iw >= w) continue;
                best = fmaxf(best, ld(x + (((size_t)img * h + ih) * w + iw) * c + ch));
            }
        }
        y[i] = cvt<T>(best);
    }
}

// Gather form: every input element looks at the windows that contain it and takes the gradient of
// those in which it is the first maximum (row-major window order).
template <typename T>
__global__ void maxpool_bwd_kernel(const T* x, const T* dy, T* dx, int n, int h, int w,
                                   int c, int ho, int wo, int k, int stride, int pad) {
    previous_grid_done();
    next_grid_may_start();
    int64_t total = (int64_t)n * h * w * c;
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < total; i += (int64_t)gridDim.x * blockDim.x) {
        int ch = (int)(i % c);
        int64_t t = i / c;
        int iw = (int)(t % w); t /= w;
        int ih = (int)(t % h);
        int img = (int)(t / h);
        const float mine = ld(x + i);
        float acc = 0.f;
        int oh_lo = max(0, (ih + pad - k + stride) / stride), oh_hi = min(ho - 1, (ih + pad) / stride);
        int ow_lo = max(0, (iw + pad - k + stride) / stride), ow_hi = min(wo - 1, (iw + pad) / stride);
        for (int oh = oh_lo; oh <= oh_hi; ++oh) {
            for (int ow = ow_lo; ow <= ow_hi; ++ow) {
                // am I the first maximum of window (oh, ow)?
                bool first = true;
                for (int r = 0; r < k && first; ++r) {
                    int yy = oh * stride - pad + r;
                    if (yy < 0 || yy >= h) continue;
                    for (int s = 0; s < k; ++s) {
                        int xx = ow * stride - pad + s;
                        if (xx < 0 || xx >= w) continue;
                        float v = ld(x + (((size_t)img * h + yy) * w + xx) * c + ch);
                        bool before = (yy < ih) || (yy == ih && xx < iw);
                        if (v > mine || (before && v == mine)) { first = false; break; }
                    }
                }
                if (first) acc += ld(dy + (((size_t)img * ho + oh) * wo + ow) * c + ch);
            }
        }
        dx[i] = cvt<T>(acc);
    }
}

// 2x2 / stride 2 / no padding on even-sized images, VEC channels per thread (16-byte accesses):
// the layout every pooling layer of the benchmark chains has.  One thread per output pixel group.
// Optional pending activation of the producer: value = round_T(max(v*scale + shift, 0)), exactly what a
// materialised copy of the activated tensor would hold.
template <typename T, int VEC>
__device__ __forceinline__ void pending_act(float (&v)[VEC], const float* act, int c, int ch) {
    if (!act) return;
#pragma unroll
    for (int k = 0; k < VEC; ++k) v[k] = (float)cvt<T>(fmaxf(fmaf(v[k], act[2 * c + ch + k], act[3 * c + ch + k]), 0.f));
}

template <typename T, int VEC>
__global__ void __launch_bounds__(256) maxpool2x2_fwd_kernel(const T* x, T* y, int64_t items, int wo, int ho, int cv, int c,
                                                             const float* act) {
    previous_grid_done();
    next_grid_may_start();
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < items; i += (int64_t)gridDim.x * blockDim.x) {
        const int cg = (int)(i % cv);
        int64_t t = i / cv;
        const int ow = (int)(t % wo); t /= wo;
        const int oh = (int)(t % ho);
        const int64_t img = t / ho;
        const T* p = x + (((img * (2 * ho) + 2 * oh) * (int64_t)(2 * wo) + 2 * ow) * c + cg * VEC);
        float a[VEC], b[VEC], d[VEC], e[VEC], o[VEC];
        load_vec<T, VEC>(p, a);
        load_vec<T, VEC>(p + c, b);
        load_vec<T, VEC>(p + (int64_t)2 * wo * c, d);
        load_vec<T, VEC>(p + (int64_t)2 * wo * c + c, e);
        pending_act<T, VEC>(a, act, c, cg * VEC); pending_act<T, VEC>(b, act, c, cg * VEC);
        pending_act<T, VEC>(d, act, c, cg * VEC); pending_act<T, VEC>(e, act, c, cg * VEC);
#pragma unroll
        for (int k = 0; k < VEC; ++k) o[k] = fmaxf(fmaxf(a[k], b[k]), fmaxf(d[k], e[k]));
        store_vec<T, VEC>(y + i * VEC, o);
    }
}

// Backward of the same: the first maximum of the window in row-major order takes the gradient.
template <typename T, int VEC>
__global__ void __launch_bounds__(256) maxpool2x2_bwd_kernel(const T* x, const T* dy, T* dx,
                                                             int64_t items, int wo, int ho, int cv, int c, const float* act) {
    previous_grid_done();
    next_grid_may_start();
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < items; i += (int64_t)gridDim.x * blockDim.x) {
        const int cg = (int)(i % cv);
        int64_t t = i / cv;
        const int ow = (int)(t % wo); t /= wo;
        const int oh = (int)(t % ho);
        const int64_t img = t / ho;
        const int64_t off = ((img * (2 * ho) + 2 * oh) * (int64_t)(2 * wo) + 2 * ow) * c + cg * VEC;
        const int64_t down = (int64_t)2 * wo * c;
        float a[VEC], b[VEC], d[VEC], e[VEC], g[VEC], oa[VEC], ob[VEC], od[VEC], oe[VEC];
        load_vec<T, VEC>(x + off, a);
        load_vec<T, VEC>(x + off + c, b);
        load_vec<T, VEC>(x + off + down, d);
        load_vec<T, VEC>(x + off + down + c, e);
        load_vec<T, VEC>(dy + i * VEC, g);
        pending_act<T, VEC>(a, act, c, cg * VEC); pending_act<T, VEC>(b, act, c, cg * VEC);
        pending_act<T, VEC>(d, act, c, cg * VEC); pending_act<T, VEC>(e, act, c, cg * VEC);
#pragma unroll
        for (int k = 0; k < VEC; ++k) {
            const float m = fmaxf(fmaxf(a[k], b[k]), fmaxf(d[k], e[k]));
            const bool ta = a[k] == m, tb = !ta && b[k] == m, td = !ta && !tb && d[k] == m, te = !ta && !tb && !td;
            oa[k] = ta ? g[k] : 0.f; ob[k] = tb ? g[k] : 0.f; od[k] = td ? g[k] : 0.f; oe[k] = te ? g[k] : 0.f;
        }
        store_vec<T, VEC>(dx + off, oa);
        store_vec<T, VEC>(dx + off + c, ob);
        store_vec<T, VEC>(dx + off + down, od);
        store_vec<T, VEC>(dx + off + down + c, oe);
    }
}

// Backward of a 2x2 pooling together with the batch-norm backward of the convolution whose output it reads through the
// pending normalisation.  The gradient between the two is a quarter of values of dy and three quarters of zeros: both passes
// route dy again from the window's four raw values instead of writing and reading that tensor (3.5 passes over z instead of
// 5.25; first the sums of g and g*z, then dz = scale*g - A - z*B).  HBM bound: 64 images of 224 x 224 x 64 390 -> 261 us with
// the finalisation between them (the second pass at 6.1 TB/s), 128 of 32 x 32 x 64 29.6 -> 19.8, 128 of 2 x 2 x 512 11.0 -> 10.5.
// The few blocks of the sums add many windows each: sums are two floats from a thread's on, also where they leave the block,
// so that only two windows are ever added in one (error of dgamma against float64, in 1e-8 of its norm, plain chains -> this: 64
// images of 56 x 56 x 256 5.1 -> 2.6, 128 of 32 x 32 x 64 5.4 -> 2.5, of which 2.5 is the rounding of the result; us of the
// pass, replayed: 28.7 -> 30.4 and 7.2 -> 7.1).
// Every thread keeps one channel group; a block has as many windows side by side as groups fit into 256 threads, and U windows in
// flight per thread (five 16-byte loads each).
//
// One channel (float) or two (bf16, packed) of a window: the activated values as the pooling saw them, the first maximum in row-major
// order takes dy, and the producer's ReLU lets it pass where that maximum is positive.  Packed, every step after the
// normalisation is one instruction for two channels (value by value the sums of VGG-16's five poolings
// took 365 us together where they take 217: issue slots).
template <typename T> struct Word;                 // 32 bits of a tensor
template <> struct Word<float> {
    static constexpr int channels = 1;
    static __device__ __forceinline__ float value(uint32_t w, int) { return __uint_as_float(w); }
    static __device__ __forceinline__ uint32_t pack(const float (&v)[1]) { return __float_as_uint(v[0]); }
    static __device__ __forceinline__ uint32_t max(uint32_t a, uint32_t b) { return __float_as_uint(fmaxf(__uint_as_float(a), __uint_as_float(b))); }
    static __device__ __forceinline__ uint32_t equal(uint32_t a, uint32_t b) { return __uint_as_float(a) == __uint_as_float(b) ? ~0u : 0u; }
    static __device__ __forceinline__ uint32_t above(uint32_t a, uint32_t b) { return __uint_as_float(a) > __uint_as_float(b) ? ~0u : 0u; }
};
template <> struct Word<__nv_bfloat16> {
    static constexpr int channels = 2;
    static __device__ __forceinline__ float value(uint32_t w, int i) { return __uint_as_float(i ? w & 0xffff0000u : w << 16); }
    static __device__ __forceinline__ __nv_bfloat162 pair(uint32_t w) { return *reinterpret_cast<__nv_bfloat162*>(&w); }
    static __device__ __forceinline__ uint32_t bits(__nv_bfloat162 p) { return *reinterpret_cast<uint32_t*>(&p); }
    static __device__ __forceinline__ uint32_t pack(const float (&v)[2]) { return bits(__floats2bfloat162_rn(v[0], v[1])); }
    static __device__ __forceinline__ uint32_t max(uint32_t a, uint32_t b) { return bits(__hmax2(pair(a), pair(b))); }
    static __device__ __forceinline__ uint32_t equal(uint32_t a, uint32_t b) { return __heq2_mask(pair(a), pair(b)); }
    static __device__ __forceinline__ uint32_t above(uint32_t a, uint32_t b) { return __hgt2_mask(pair(a), pair(b)); }
};
// z: a word of each of the window's pixels, as values and as bits; returns dy's word where it passes, take[q]: where pixel q gets it
template <typename T>
__device__ __forceinline__ uint32_t route_2x2(const float (&z)[4][Word<T>::channels], uint32_t g, const float* sc, const float* sh, uint32_t (&take)[4]) {
    using W = Word<T>;
    uint32_t a[4];
#pragma unroll
    for (int q = 0; q < 4; ++q) {
        float v[W::channels];
#pragma unroll
        for (int i = 0; i < W::channels; ++i) v[i] = fmaf(z[q][i], sc[i], sh[i]);
        a[q] = W::max(W::pack(v), 0u);
    }
    const uint32_t m = W::max(W::max(a[0], a[1]), W::max(a[2], a[3]));
    take[0] = W::equal(a[0], m);
    take[1] = W::equal(a[1], m) & ~take[0];
    take[2] = W::equal(a[2], m) & ~(take[0] | take[1]);
    take[3] = ~(take[0] | take[1] | take[2]);
    return g & W::above(m, 0u);
}
struct PoolBn {
    int64_t windows;
    int wo, c, groups, across;         // groups = c / VEC; across = windows side by side in a block
};
constexpr int kPoolBnU = 2;
// five vectors of a window: its four pixels and dy
template <typename T, int VEC>
struct PoolWindow {
    uint32_t z[4][4], g[4];
    int64_t off;
    static __device__ __forceinline__ void fetch(uint32_t (&d)[4], const T* p) {
        const uint4 q = *reinterpret_cast<const uint4*>(p);
        d[0] = q.x; d[1] = q.y; d[2] = q.z; d[3] = q.w;
    }
    // window w = (image and row) * wo + column: its first pixel is 4 w - 2 column
    __device__ __forceinline__ void load(const PoolBn& p, const T* zp, const T* dy, uint32_t w, int ch) {
        off = ((int64_t)4 * w - 2 * (int64_t)(w % (uint32_t)p.wo)) * p.c + ch;
        const int64_t down = (int64_t)2 * p.wo * p.c;
        fetch(z[0], zp + off); fetch(z[1], zp + off + p.c); fetch(z[2], zp + off + down); fetch(z[3], zp + off + down + p.c);
        fetch(g, dy + (int64_t)w * p.c + ch);
    }
};
template <typename T, int VEC>
__global__ void __launch_bounds__(256, 2) maxpool2x2_bn_sums_kernel(const T* z, const T* dy, const float* stats, PoolBn p, float* partial) {
    previous_grid_done();
    next_grid_may_start();
    using W = Word<T>;
    constexpr int U = kPoolBnU, C = W::channels;
    __shared__ float2 red[256][2 * VEC + 1], few[256];
    const int group = threadIdx.x % p.groups, row = threadIdx.x / p.groups, ch = group * VEC;
    float2 s0[VEC], s1[VEC];
    float sc[VEC], sh[VEC];
#pragma unroll
    for (int k = 0; k < VEC; ++k) { sc[k] = stats[2 * p.c + ch + k]; sh[k] = stats[3 * p.c + ch + k]; s0[k] = s1[k] = make_float2(0.f, 0.f); }
    const int64_t hop = (int64_t)gridDim.x * p.across;
    if (row < p.across) {
        for (int64_t w0 = (int64_t)blockIdx.x * p.across + row; w0 < p.windows; w0 += U * hop) {
            PoolWindow<T, VEC> win[U];
#pragma unroll
            for (int u = 0; u < U; ++u)
                if (w0 + u * hop < p.windows) win[u].load(p, z, dy, (uint32_t)(w0 + u * hop), ch);
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                // (the windows of a step join the running sums, two floats each, one by one in float32; in bfloat16, whose products
                // are exact and values few bits, added up)
                float t0[C], t1[C];
#pragma unroll
                for (int i = 0; i < C; ++i) t0[i] = t1[i] = 0.f;
#pragma unroll
                for (int u = 0; u < U; ++u) {
                    if (w0 + u * hop >= p.windows) break;
                    float v[4][C];
                    uint32_t take[4], at = 0u;
#pragma unroll
                    for (int q = 0; q < 4; ++q)
#pragma unroll
                        for (int i = 0; i < C; ++i) v[q][i] = W::value(win[u].z[q][j], i);
                    const uint32_t g = route_2x2<T>(v, win[u].g[j], sc + j * C, sh + j * C, take);
                    // one of the four has the gradient: its z is the only one that counts
#pragma unroll
                    for (int q = 0; q < 4; ++q) at |= win[u].z[q][j] & take[q];
#pragma unroll
                    for (int i = 0; i < C; ++i) {
                        t0[i] += W::value(g, i); t1[i] = fmaf(W::value(g, i), W::value(at, i), t1[i]);
                        if (C == 1) { carry_sum(s0[j * C + i], t0[i]); carry_sum(s1[j * C + i], t1[i]); t0[i] = t1[i] = 0.f; }
                    }
                }
                if (C > 1) {
#pragma unroll
                    for (int i = 0; i < C; ++i) { carry_sum(s0[j * C + i], t0[i]); carry_sum(s1[j * C + i], t1[i]); }
                }
            }
        }
    }
#pragma unroll
    for (int k = 0; k < VEC; ++k) { red[threadIdx.x][k] = s0[k]; red[threadIdx.x][VEC + k] = s1[k]; }
    __syncthreads();
    // a thread or a few per column (channel group, sum) add up its rows, and one of them the few; both floats of a sum leave, as
    // rows of their own
    const int columns = 2 * VEC * p.groups, share = max(1, 256 / columns);
    auto leave = [&](int col, float2 sum) {
        const int k = col % (2 * VEC);
        float* const to = partial + ((size_t)blockIdx.x * 4 + k / VEC) * p.c + col / (2 * VEC) * VEC + k % VEC;
        to[0] = sum.x;
        to[2 * p.c] = sum.y;
    };
    for (int i = threadIdx.x; i < columns * share; i += 256) {
        const int col = i % columns, part = i / columns;
        float2 sum[2] = {make_float2(0.f, 0.f), make_float2(0.f, 0.f)};
        for (int r = part; r < p.across; r += 4 * share) {
            float2 v[4];
#pragma unroll
            for (int u = 0; u < 4; ++u) v[u] = r + u * share < p.across ? red[(r + u * share) * p.groups + col / (2 * VEC)][col % (2 * VEC)] : make_float2(0.f, 0.f);
#pragma unroll
            for (int u = 0; u < 4; ++u) { two_sum(sum[u & 1], v[u].x); sum[u & 1].y += v[u].y; }
        }
        two_sum(sum[0], sum[1].x); sum[0].y += sum[1].y;
        if (share == 1) leave(col, sum[0]);
        else few[i] = sum[0];
    }
    if (share == 1) return;
    __syncthreads();
    if ((int)threadIdx.x < columns) {
        float2 sum = few[threadIdx.x];
        for (int part = 1; part < share; ++part) { const float2 v = few[part * columns + threadIdx.x]; two_sum(sum, v.x); sum.y += v.y; }
        leave(threadIdx.x, sum);
    }
}
template <typename T, int VEC>
__global__ void __launch_bounds__(256, 2) maxpool2x2_bn_apply_kernel(const T* z, const T* dy, const float* stats, const float* coef, PoolBn p, T* dz) {
    previous_grid_done();
    next_grid_may_start();
    using W = Word<T>;
    constexpr int U = kPoolBnU, C = W::channels;
    const int group = threadIdx.x % p.groups, row = threadIdx.x / p.groups, ch = group * VEC;
    if (row >= p.across) return;
    const int64_t w0 = (int64_t)blockIdx.x * p.across * U + row;
    PoolWindow<T, VEC> win[U];
#pragma unroll
    for (int u = 0; u < U; ++u)
        if (w0 + u * p.across < p.windows) win[u].load(p, z, dy, (uint32_t)(w0 + u * p.across), ch);
    float sc[VEC], sh[VEC], ca[VEC], cb[VEC];
#pragma unroll
    for (int k = 0; k < VEC; ++k) { sc[k] = stats[2 * p.c + ch + k]; sh[k] = stats[3 * p.c + ch + k]; ca[k] = coef[ch + k]; cb[k] = coef[p.c + ch + k]; }
#pragma unroll
    for (int u = 0; u < U; ++u) {
        if (w0 + u * p.across >= p.windows) break;
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            float v[4][C];
            uint32_t take[4];
#pragma unroll
            for (int q = 0; q < 4; ++q)
#pragma unroll
                for (int i = 0; i < C; ++i) v[q][i] = W::value(win[u].z[q][j], i);
            const uint32_t g = route_2x2<T>(v, win[u].g[j], sc + j * C, sh + j * C, take);
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                float o[C];
#pragma unroll
                for (int i = 0; i < C; ++i) o[i] = fmaf(-v[q][i], cb[j * C + i], fmaf(sc[j * C + i], W::value(g & take[q], i), -ca[j * C + i]));
                win[u].z[q][j] = W::pack(o);
            }
        }
        const int64_t down = (int64_t)2 * p.wo * p.c;
        auto leave = [&](T* to, const uint32_t (&d)[4]) { *reinterpret_cast<uint4*>(to) = make_uint4(d[0], d[1], d[2], d[3]); };
        leave(dz + win[u].off, win[u].z[0]);
        leave(dz + win[u].off + p.c, win[u].z[1]);
        leave(dz + win[u].off + down, win[u].z[2]);
        leave(dz + win[u].off + down + p.c, win[u].z[3]);
    }
}

// Forward, optionally through the pending normalisation, in the same shape (value by value, with the coefficients read again for
// every window: 107 us for 64 images of 224 x 224 x 64, this 80).
template <typename T, int VEC, bool ACT>
__global__ void __launch_bounds__(256, 3) maxpool2x2_windows_kernel(const T* z, const float* stats, PoolBn p, T* y) {
    previous_grid_done();
    next_grid_may_start();
    using W = Word<T>;
    constexpr int U = kPoolBnU, C = W::channels;
    const int group = threadIdx.x % p.groups, row = threadIdx.x / p.groups, ch = group * VEC;
    if (row >= p.across) return;
    const int64_t w0 = (int64_t)blockIdx.x * p.across * U + row, down = (int64_t)2 * p.wo * p.c;
    uint4 q[U][4];
#pragma unroll
    for (int u = 0; u < U; ++u) {
        const int64_t w = w0 + u * p.across;
        if (w >= p.windows) break;
        const T* const at = z + (4 * w - 2 * (int64_t)((uint32_t)w % (uint32_t)p.wo)) * p.c + ch;
        q[u][0] = *reinterpret_cast<const uint4*>(at); q[u][1] = *reinterpret_cast<const uint4*>(at + p.c);
        q[u][2] = *reinterpret_cast<const uint4*>(at + down); q[u][3] = *reinterpret_cast<const uint4*>(at + down + p.c);
    }
    float sc[VEC], sh[VEC];
#pragma unroll
    for (int k = 0; k < VEC; ++k) { sc[k] = ACT ? stats[2 * p.c + ch + k] : 1.f; sh[k] = ACT ? stats[3 * p.c + ch + k] : 0.f; }
#pragma unroll
    for (int u = 0; u < U; ++u) {
        const int64_t w = w0 + u * p.across;
        if (w >= p.windows) break;
        uint32_t out[4];
#pragma unroll
        for (int j = 0; j < 4; ++j) {
#pragma unroll
            for (int e = 0; e < 4; ++e) {
                uint32_t word = j == 0 ? q[u][e].x : j == 1 ? q[u][e].y : j == 2 ? q[u][e].z : q[u][e].w;
                if (ACT) {
                    float v[C];
#pragma unroll
                    for (int i = 0; i < C; ++i) v[i] = fmaf(W::value(word, i), sc[j * C + i], sh[j * C + i]);
                    word = W::pack(v);
                }
                out[j] = e > 0 ? W::max(out[j], word) : ACT ? W::max(word, 0u) : word;         // (0: the ReLU)
            }
        }
        *reinterpret_cast<uint4*>(y + w * p.c + ch) = make_uint4(out[0], out[1], out[2], out[3]);
    }
}

static bool pool_2x2(int dtype, int h, int w, int c, int k, int stride, int pad) {
    const int vec = dtype == CKPT_DTYPE_BF16 ? 8 : 4;
    return k == 2 && stride == 2 && pad == 0 && h % 2 == 0 && w % 2 == 0 && c % vec == 0;
}
// The residual networks' 3x3 pooling with stride 2 and padding 1 behind the stem.
static bool pool_3x3(int dtype, int c, int k, int stride, int pad) {
    return dtype == CKPT_DTYPE_BF16 && k == 3 && stride == 2 && pad == 1 && c % 8 == 0 && c <= 1024 && 256 % (c / 8) == 0;
}
bool maxpool_fuses_activation(int dtype, int h, int w, int c, int k, int stride, int pad) {
    return pool_2x2(dtype, h, w, c, k, stride, pad) || pool_3x3(dtype, c, k, stride, pad);
}

// 3x3 pooling, stride 2, padding 1, of a pre-normalisation tensor: what is pooled is bf16(max(z*scale + shift, 0)), which
// grows with z where the scale is positive and falls where it is negative, so the forward takes the maximum of z (its sign
// flipped for negative scales) in packed pairs and normalises nine times less.  A thread owns eight channels of a window,
// its nine loads in flight at once.
__device__ __forceinline__ void pool3_load(const __nv_bfloat16* z, int64_t img, int oh, int ow, int h, int w, int c, int ch, uint4 (&r)[9], uint32_t& valid) {
    valid = 0u;
#pragma unroll
    for (int t = 0; t < 9; ++t) {
        const int ih = 2 * oh - 1 + t / 3, iw = 2 * ow - 1 + t % 3;
        if (ih >= 0 && ih < h && iw >= 0 && iw < w) {
            r[t] = *reinterpret_cast<const uint4*>(z + ((img * h + ih) * w + iw) * c + ch);
            valid |= 1u << t;
        }
    }
}
__device__ __forceinline__ uint32_t& word(uint4& v, int k) { return k == 0 ? v.x : k == 1 ? v.y : k == 2 ? v.z : v.w; }
__global__ void __launch_bounds__(256) maxpool3_fwd_act_kernel(const __nv_bfloat16* z, __nv_bfloat16* y, int64_t items, int h, int w,
                                                               int c, int ho, int wo, const float* act) {
    previous_grid_done();
    next_grid_may_start();
    const int lanes = c / 8;
    const int ch = (int)(threadIdx.x % lanes) * 8;              // 256 and the grid stride are multiples of `lanes`
    float sc[8], sh[8];
    uint32_t flip[4];
#pragma unroll
    for (int k = 0; k < 8; ++k) { sc[k] = act[2 * c + ch + k]; sh[k] = act[3 * c + ch + k]; }
#pragma unroll
    for (int k = 0; k < 4; ++k) flip[k] = (sc[2 * k] < 0.f ? 0x8000u : 0u) | (sc[2 * k + 1] < 0.f ? 0x80000000u : 0u);
    for (int64_t i = (int64_t)blockIdx.x * 256 + threadIdx.x; i < items; i += (int64_t)gridDim.x * 256) {
        const uint32_t t = (uint32_t)(i / lanes);
        const int ow = (int)(t % (uint32_t)wo), oh = (int)(t / (uint32_t)wo % (uint32_t)ho);
        const int64_t img = t / ((uint32_t)wo * (uint32_t)ho);
        uint4 r[9];
        uint32_t valid;
        pool3_load(z, img, oh, ow, h, w, c, ch, r, valid);
        uint4 best = make_uint4(0xff80ff80u, 0xff80ff80u, 0xff80ff80u, 0xff80ff80u);      // -infinity
#pragma unroll
        for (int q = 0; q < 9; ++q) {
            if (!((valid >> q) & 1u)) continue;
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                const uint32_t v = word(r[q], k) ^ flip[k];
                const __nv_bfloat162 m = __hmax2(*reinterpret_cast<const __nv_bfloat162*>(&word(best, k)), *reinterpret_cast<const __nv_bfloat162*>(&v));
                word(best, k) = *reinterpret_cast<const uint32_t*>(&m);
            }
        }
        float o[8];
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            const uint32_t v = word(best, k) ^ flip[k];
            o[2 * k] = fmaxf(fmaf(__uint_as_float(v << 16), sc[2 * k], sh[2 * k]), 0.f);
            o[2 * k + 1] = fmaxf(fmaf(__uint_as_float(v & 0xffff0000u), sc[2 * k + 1], sh[2 * k + 1]), 0.f);
        }
        store_vec<__nv_bfloat16, 8>(y + i * 8, o);
    }
}
// Position (0..8) of the first maximum of the normalised values, one byte per channel.
__global__ void __launch_bounds__(256) maxpool3_arg_act_kernel(const __nv_bfloat16* z, uint8_t* arg, int64_t items, int h, int w,
                                                               int c, int ho, int wo, const float* act) {
    previous_grid_done();
    next_grid_may_start();
    const int lanes = c / 8;
    const int ch = (int)(threadIdx.x % lanes) * 8;
    float sc[8], sh[8];
#pragma unroll
    for (int k = 0; k < 8; ++k) { sc[k] = act[2 * c + ch + k]; sh[k] = act[3 * c + ch + k]; }
    for (int64_t i = (int64_t)blockIdx.x * 256 + threadIdx.x; i < items; i += (int64_t)gridDim.x * 256) {
        const uint32_t t = (uint32_t)(i / lanes);
        const int ow = (int)(t % (uint32_t)wo), oh = (int)(t / (uint32_t)wo % (uint32_t)ho);
        const int64_t img = t / ((uint32_t)wo * (uint32_t)ho);
        uint4 r[9];
        uint32_t valid;
        pool3_load(z, img, oh, ow, h, w, c, ch, r, valid);
        uint4 best = make_uint4(0xbf80bf80u, 0xbf80bf80u, 0xbf80bf80u, 0xbf80bf80u);      // -1: below every normalised value
        uint4 pos = make_uint4(0u, 0u, 0u, 0u);
#pragma unroll
        for (int q = 0; q < 9; ++q) {
            if (!((valid >> q) & 1u)) continue;
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                const uint32_t v = word(r[q], k);
                const __nv_bfloat162 a = __floats2bfloat162_rn(fmaxf(fmaf(__uint_as_float(v << 16), sc[2 * k], sh[2 * k]), 0.f),
                                                               fmaxf(fmaf(__uint_as_float(v & 0xffff0000u), sc[2 * k + 1], sh[2 * k + 1]), 0.f));
                const __nv_bfloat162 b = *reinterpret_cast<const __nv_bfloat162*>(&word(best, k));
                const uint32_t more = __hgt2_mask(a, b);                                  // strict: the first maximum stays
                word(pos, k) = (word(pos, k) & ~more) | ((uint32_t)(q * 0x10001) & more);
                const __nv_bfloat162 m = __hmax2(a, b);
                word(best, k) = *reinterpret_cast<const uint32_t*>(&m);
            }
        }
        *reinterpret_cast<uint2*>(arg + i * 8) = make_uint2(__byte_perm(pos.x, pos.y, 0x6420), __byte_perm(pos.z, pos.w, 0x6420));
    }
}
// Gradient of a 2 x 2 quad of inputs (rows 2a, 2a + 1; columns 2b, 2b + 1) from the recorded positions: an even row belongs
// to window a only (its middle row), an odd one to windows a (last row) and a + 1 (first row).  With `act` the producer's
// batch-norm backward sums (sum g, sum g*z over the values its ReLU passes) go to `partial`, a row pair per block.
template <bool SUMS>
__global__ void __launch_bounds__(256) maxpool3_bwd_kernel(const uint8_t* arg, const __nv_bfloat16* dy, __nv_bfloat16* dx,
                                                           int64_t items, int h, int w, int c, int ho, int wo, const __nv_bfloat16* z,
                                                           const float* act, float* partial) {
    previous_grid_done();
    next_grid_may_start();
    __shared__ float red[SUMS ? 256 : 1][17];
    const int lanes = c / 8;
    const int ch = (int)(threadIdx.x % lanes) * 8;
    float sc[8], sh[8], s0[8], s1[8];
#pragma unroll
    for (int k = 0; k < 8; ++k) { sc[k] = SUMS ? act[2 * c + ch + k] : 0.f; sh[k] = SUMS ? act[3 * c + ch + k] : 0.f; s0[k] = 0.f; s1[k] = 0.f; }
    for (int64_t i = (int64_t)blockIdx.x * 256 + threadIdx.x; i < items; i += (int64_t)gridDim.x * 256) {
        const uint32_t t = (uint32_t)(i / lanes);
        const int b = (int)(t % (uint32_t)wo), a = (int)(t / (uint32_t)wo % (uint32_t)ho);
        const int64_t img = t / ((uint32_t)wo * (uint32_t)ho);
        uint2 pos[4];
        uint4 raw[4], zr[4];
#pragma unroll
        for (int q = 0; q < 4; ++q) {                            // windows (a + q/2, b + q%2)
            const bool in = a + q / 2 < ho && b + q % 2 < wo;
            const int64_t o = ((img * ho + a + q / 2) * wo + b + q % 2) * c + ch;
            pos[q] = in ? *reinterpret_cast<const uint2*>(arg + o) : make_uint2(0xffffffffu, 0xffffffffu);
            raw[q] = in ? *reinterpret_cast<const uint4*>(dy + o) : make_uint4(0u, 0u, 0u, 0u);
        }
#pragma unroll
        for (int q = 0; q < 4; ++q)
            if (SUMS && 2 * a + q / 2 < h && 2 * b + q % 2 < w)
                zr[q] = *reinterpret_cast<const uint4*>(z + ((img * h + 2 * a + q / 2) * w + 2 * b + q % 2) * c + ch);
        float g[4][8];
#pragma unroll
        for (int q = 0; q < 4; ++q) unpack<__nv_bfloat16, 8>(from_uint4<__nv_bfloat16, 8>(raw[q]), g[q]);
        auto at = [&](int q, int k) { return (int)((k < 4 ? pos[q].x >> (8 * k) : pos[q].y >> (8 * (k - 4))) & 0xffu); };
#pragma unroll
        for (int in = 0; in < 4; ++in) {
            if (2 * a + in / 2 >= h || 2 * b + in % 2 >= w) continue;
            float o[8];
#pragma unroll
            for (int k = 0; k < 8; ++k) {
                o[k] = 0.f;
#pragma unroll
                for (int q = 0; q < 4; ++q) {
                    if (q / 2 > in / 2 || q % 2 > in % 2) continue;                      // an even row or column has one window
                    const int r = in / 2 ? (q / 2 ? 0 : 2) : 1, s = in % 2 ? (q % 2 ? 0 : 2) : 1;
                    o[k] += at(q, k) == r * 3 + s ? g[q][k] : 0.f;
                }
            }
            const uint4 packed = as_uint4(pack_raw<__nv_bfloat16, 8>(o));
            *reinterpret_cast<uint4*>(dx + ((img * h + 2 * a + in / 2) * w + 2 * b + in % 2) * c + ch) = packed;
            if (SUMS) {
                float v[8], stored[8];
                unpack<__nv_bfloat16, 8>(from_uint4<__nv_bfloat16, 8>(zr[in]), v);
                unpack<__nv_bfloat16, 8>(from_uint4<__nv_bfloat16, 8>(packed), stored);
#pragma unroll
                for (int k = 0; k < 8; ++k)
                    if (fmaf(v[k], sc[k], sh[k]) > 0x1p-134f) { s0[k] += stored[k]; s1[k] = fmaf(stored[k], v[k], s1[k]); }
            }
        }
    }
    if (!SUMS) return;
#pragma unroll
    for (int k = 0; k < 8; ++k) { red[threadIdx.x][k] = s0[k]; red[threadIdx.x][8 + k] = s1[k]; }
    __syncthreads();
    for (int off = 128; off >= lanes; off >>= 1) {               // `lanes` divides 256: threads t and t + off hold the same group
        if ((int)threadIdx.x < off)
#pragma unroll
            for (int k = 0; k < 16; ++k) red[threadIdx.x][k] += red[threadIdx.x + off][k];
        __syncthreads();
    }
    if ((int)threadIdx.x < lanes) {
#pragma unroll
        for (int k = 0; k < 8; ++k) {
            partial[((size_t)blockIdx.x * 2 + 0) * c + ch + k] = red[threadIdx.x][k];
            partial[((size_t)blockIdx.x * 2 + 1) * c + ch + k] = red[threadIdx.x][8 + k];
        }
    }
}

// Vector forms of the two general pooling kernels: one thread handles VEC consecutive channels of a
// pixel with 16-byte accesses; same window order and tie rule as the scalar kernels.
template <typename T, int VEC>
__global__ void __launch_bounds__(256) maxpool_fwd_vec_kernel(const T* x, T* y, int64_t items, int h, int w,
                                                              int c, int ho, int wo, int k, int stride, int pad) {
    previous_grid_done();
    next_grid_may_start();
    const int lanes = c / VEC;
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < items; i += (int64_t)gridDim.x * blockDim.x) {
        const int ch = (int)(i % lanes) * VEC;
        int64_t t = i / lanes;
        const int ow = (int)(t % wo); t /= wo;
        const int oh = (int)(t % ho);
        const int64_t img = t / ho;
        float best[VEC];
#pragma unroll
        for (int e = 0; e < VEC; ++e) best[e] = -INFINITY;
        for (int r = 0; r < k; ++r) {
            const int ih = oh * stride - pad + r;
            if (ih < 0 || ih >= h) continue;
            for (int q = 0; q < k; ++q) {
                const int iw = ow * stride - pad + q;
                if (iw < 0 || iw >= w) continue;
                float v[VEC];
                load_vec<T, VEC>(x + ((img * h + ih) * w + iw) * c + ch, v);
#pragma unroll
                for (int e = 0; e < VEC; ++e) best[e] = fmaxf(best[e], v[e]);
            }
        }
        store_vec<T, VEC>(y + i * VEC, best);
    }
}

template <typename T, int VEC>
__global__ void __launch_bounds__(256) maxpool_bwd_vec_kernel(const T* x, const T* dy, T* dx,
                                                              int64_t items, int h, int w, int c, int ho, int wo, int k, int stride,
                                                              int pad) {
    previous_grid_done();
    next_grid_may_start();
    const int lanes = c / VEC;
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < items; i += (int64_t)gridDim.x * blockDim.x) {
        const int ch = (int)(i % lanes) * VEC;
        int64_t t = i / lanes;
        const int iw = (int)(t % w); t /= w;
        const int ih = (int)(t % h);
        const int64_t img = t / h;
        float mine[VEC], acc[VEC];
        load_vec<T, VEC>(x + i * VEC, mine);
#pragma unroll
        for (int e = 0; e < VEC; ++e) acc[e] = 0.f;
        const int oh_lo = max(0, (ih + pad - k + stride) / stride), oh_hi = min(ho - 1, (ih + pad) / stride);
        const int ow_lo = max(0, (iw + pad - k + stride) / stride), ow_hi = min(wo - 1, (iw + pad) / stride);
        for (int oh = oh_lo; oh <= oh_hi; ++oh) {
            for (int ow = ow_lo; ow <= ow_hi; ++ow) {
                // in which channels am I the first maximum of window (oh, ow)?
                bool first[VEC];
#pragma unroll
                for (int e = 0; e < VEC; ++e) first[e] = true;
                for (int r = 0; r < k; ++r) {
                    const int yy = oh * stride - pad + r;
                    if (yy < 0 || yy >= h) continue;
                    for (int q = 0; q < k; ++q) {
                        const int xx = ow * stride - pad + q;
                        if (xx < 0 || xx >= w || (yy == ih && xx == iw)) continue;
                        float v[VEC];
                        load_vec<T, VEC>(x + ((img * h + yy) * w + xx) * c + ch, v);
                        const bool before = (yy < ih) || (yy == ih && xx < iw);
#pragma unroll
                        for (int e = 0; e < VEC; ++e)
                            if (v[e] > mine[e] || (before && v[e] == mine[e])) first[e] = false;
                    }
                }
                float g[VEC];
                load_vec<T, VEC>(dy + ((img * ho + oh) * wo + ow) * c + ch, g);
#pragma unroll
                for (int e = 0; e < VEC; ++e) acc[e] += first[e] ? g[e] : 0.f;
            }
        }
        store_vec<T, VEC>(dx + i * VEC, acc);
    }
}

// General pooling backward in two passes when scratch is available.  Pass 1, one thread per window and VEC
// channels: the position (r*k + q) of the first maximum, one byte per channel.  Pass 2, one thread per input
// pixel and VEC channels: for each of the (at most ceil(k/stride)^2) windows that contain the pixel, take the
// window's gradient where the recorded position is this pixel's.  Pass 2 never reads x: eight small loads per
// thread instead of re-scanning up to four whole windows.
template <typename T, int VEC>
__global__ void __launch_bounds__(256) maxpool_argmax_kernel(const T* x, uint8_t* arg, int64_t items, int h,
                                                             int w, int c, int ho, int wo, int k, int stride, int pad) {
    previous_grid_done();
    next_grid_may_start();
    const int lanes = c / VEC;
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < items; i += (int64_t)gridDim.x * blockDim.x) {
        const int ch = (int)(i % lanes) * VEC;
        int64_t t = i / lanes;
        const int ow = (int)(t % wo); t /= wo;
        const int oh = (int)(t % ho);
        const int64_t img = t / ho;
        float best[VEC];
        uint8_t pos[VEC];
#pragma unroll
        for (int e = 0; e < VEC; ++e) { best[e] = -INFINITY; pos[e] = 255; }
        for (int r = 0; r < k; ++r) {
            const int ih = oh * stride - pad + r;
            if (ih < 0 || ih >= h) continue;
            for (int q = 0; q < k; ++q) {
                const int iw = ow * stride - pad + q;
                if (iw < 0 || iw >= w) continue;
                float v[VEC];
                load_vec<T, VEC>(x + ((img * h + ih) * w + iw) * c + ch, v);
#pragma unroll
                for (int e = 0; e < VEC; ++e)
                    if (v[e] > best[e] || pos[e] == 255) { best[e] = v[e]; pos[e] = (uint8_t)(r * k + q); }   // strict: the first maximum stays
            }
        }
#pragma unroll
        for (int e = 0; e < VEC; ++e) arg[i * VEC + e] = pos[e];
    }
}

template <typename T, int VEC>
__global__ void __launch_bounds__(256) maxpool_bwd_arg_kernel(const uint8_t* arg, const T* dy, T* dx,
                                                              int64_t items, int h, int w, int c, int ho, int wo, int k, int stride,
                                                              int pad) {
    previous_grid_done();
    next_grid_may_start();
    const int lanes = c / VEC;
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < items; i += (int64_t)gridDim.x * blockDim.x) {
        const int ch = (int)(i % lanes) * VEC;
        int64_t t = i / lanes;
        const int iw = (int)(t % w); t /= w;
        const int ih = (int)(t % h);
        const int64_t img = t / h;
        float acc[VEC];
#pragma unroll
        for (int e = 0; e < VEC; ++e) acc[e] = 0.f;
        const int oh_lo = max(0, (ih + pad - k + stride) / stride), oh_hi = min(ho - 1, (ih + pad) / stride);
        const int ow_lo = max(0, (iw + pad - k + stride) / stride), ow_hi = min(wo - 1, (iw + pad) / stride);
        for (int oh = oh_lo; oh <= oh_hi; ++oh) {
            for (int ow = ow_lo; ow <= ow_hi; ++ow) {
                const int mine = (ih - (oh * stride - pad)) * k + (iw - (ow * stride - pad));
                const int64_t o = ((img * ho + oh) * wo + ow) * c + ch;
                uint8_t pos[VEC];
                if constexpr (VEC == 8) *reinterpret_cast<uint2*>(pos) = *reinterpret_cast<const uint2*>(arg + o);
                else *reinterpret_cast<uint32_t*>(pos) = *reinterpret_cast<const uint32_t*>(arg + o);
                float g[VEC];
                load_vec<T, VEC>(dy + o, g);
#pragma unroll
                for (int e = 0; e < VEC; ++e) acc[e] += pos[e] == mine ? g[e] : 0.f;
            }
        }
        store_vec<T, VEC>(dx + i * VEC, acc);
    }
}

int64_t maxpool_backward_scratch_bytes(int dtype, int n, int h, int w, int c, int k, int stride, int pad) {
    if (pool_2x2(dtype, h, w, c, k, stride, pad) || k * k > 250) return 0;
    const int vec = dtype == CKPT_DTYPE_BF16 ? 8 : 4;
    if (c % vec) return 0;
    const int ho = (h + 2 * pad - k) / stride + 1, wo = (w + 2 * pad - k) / stride + 1;
    // (behind the positions, room for the batch-norm sums of the 3x3 kernel)
    return align_up((int64_t)n * ho * wo * c, 256) + (pool_3x3(dtype, c, k, stride, pad) ? bn_scratch_bytes(0, c) : 0);
}

// (the kernels that walk windows by a 32-bit number and keep a channel group per thread)
static bool pool_2x2_windows(int dtype, int n, int h, int w, int c, const void* a, const void* b) {
    return c / (dtype == CKPT_DTYPE_BF16 ? 8 : 4) <= 256 && (int64_t)n * (h / 2) * (w / 2) < ((int64_t)1 << 31) && !(((uintptr_t)a | (uintptr_t)b) & 15u);
}
static PoolBn pool_windows(int n, int h, int w, int c, int vec) {
    PoolBn p;
    p.wo = w / 2; p.windows = (int64_t)n * (h / 2) * p.wo; p.c = c; p.groups = c / vec; p.across = 256 / p.groups;
    return p;
}
static unsigned pool_blocks(const PoolBn& p) { return (unsigned)std::max<int64_t>(1, (p.windows + p.across * kPoolBnU - 1) / (p.across * kPoolBnU)); }
int maxpool_forward(int dtype, int n, int h, int w, int c, int k, int stride, int pad, const void* x, void* y, const float* act, void* stream) {
    int ho = (h + 2 * pad - k) / stride + 1, wo = (w + 2 * pad - k) / stride + 1;
    if (pool_2x2(dtype, h, w, c, k, stride, pad)) {
        const int vec = dtype == CKPT_DTYPE_BF16 ? 8 : 4;
        if (pool_2x2_windows(dtype, n, h, w, c, x, y)) {
            const PoolBn p = pool_windows(n, h, w, c, vec);
            const unsigned blocks = pool_blocks(p);
            cudaStream_t st = (cudaStream_t)stream;
            if (dtype == CKPT_DTYPE_BF16)
                launch(Start::ON_STREAMS, act ? maxpool2x2_windows_kernel<__nv_bfloat16, 8, true> : maxpool2x2_windows_kernel<__nv_bfloat16, 8, false>, blocks, 256, 0, st,
                       (const __nv_bfloat16*)x, act, p, (__nv_bfloat16*)y);
            else
                launch(Start::ON_STREAMS, act ? maxpool2x2_windows_kernel<float, 4, true> : maxpool2x2_windows_kernel<float, 4, false>, blocks, 256, 0, st, (const float*)x, act, p, (float*)y);
            CKPT_LAUNCH_CHECK("max-pool 2x2 forward");
            return CKPT_OK;
        }
        const int64_t items = (int64_t)n * ho * wo * (c / vec);
        if (dtype == CKPT_DTYPE_BF16)
            launch(Start::ON_STREAMS, maxpool2x2_fwd_kernel<__nv_bfloat16, 8>, elementwise_grid(items), 256, 0, (cudaStream_t)stream, (const __nv_bfloat16*)x, (__nv_bfloat16*)y, items, wo, ho, c / vec, c, act);
        else
            launch(Start::ON_STREAMS, maxpool2x2_fwd_kernel<float, 4>, elementwise_grid(items), 256, 0, (cudaStream_t)stream, (const float*)x, (float*)y, items, wo, ho, c / vec, c, act);
        CKPT_LAUNCH_CHECK("max-pool 2x2 forward");
        return CKPT_OK;
    }
    if (act && pool_3x3(dtype, c, k, stride, pad)) {
        const int64_t items = (int64_t)n * ho * wo * (c / 8);
        launch(Start::ON_STREAMS, maxpool3_fwd_act_kernel, elementwise_grid(items), 256, 0, (cudaStream_t)stream, (const __nv_bfloat16*)x, (__nv_bfloat16*)y, items, h, w, c, ho, wo, act);
        CKPT_LAUNCH_CHECK("max-pool 3x3 forward");
        return CKPT_OK;
    }
    if (act) { set_error("the general pooling kernel takes an activated input"); return CKPT_E_BAD_ARG; }
    if (c % bn_vec(dtype, c) == 0 && bn_vec(dtype, c) > 1) {
        const int64_t items = (int64_t)n * ho * wo * (c / bn_vec(dtype, c));
        if (dtype == CKPT_DTYPE_BF16)
            launch(Start::ON_STREAMS, maxpool_fwd_vec_kernel<__nv_bfloat16, 8>, elementwise_grid(items), 256, 0, (cudaStream_t)stream, (const __nv_bfloat16*)x, (__nv_bfloat16*)y, items, h, w, c, ho, wo, k, stride, pad);
        else
            launch(Start::ON_STREAMS, maxpool_fwd_vec_kernel<float, 4>, elementwise_grid(items), 256, 0, (cudaStream_t)stream, (const float*)x, (float*)y, items, h, w, c, ho, wo, k, stride, pad);
        CKPT_LAUNCH_CHECK("max-pool forward");
        return CKPT_OK;
    }
    unsigned grid = elementwise_grid((int64_t)n * ho * wo * c);
    if (dtype == CKPT_DTYPE_BF16)
        launch(Start::ON_STREAMS, maxpool_fwd_kernel<__nv_bfloat16>, grid, 256, 0, (cudaStream_t)stream, (const __nv_bfloat16*)x, (__nv_bfloat16*)y, n, h, w, c, ho, wo, k, stride, pad);
    else
        launch(Start::ON_STREAMS, maxpool_fwd_kernel<float>, grid, 256, 0, (cudaStream_t)stream, (const float*)x, (float*)y, n, h, w, c, ho, wo, k, stride, pad);
    CKPT_LAUNCH_CHECK("max-pool forward");
    return CKPT_OK;
}

bool maxpool_joins_bn_backward(int dtype, int n, int h, int w, int c, int k, int stride, int pad, const void* z, const void* dy, const void* dz) {
    return pool_2x2(dtype, h, w, c, k, stride, pad) && pool_2x2_windows(dtype, n, h, w, c, z, dy) && (uintptr_t)dz % 16 == 0;
}
template <typename T, int VEC>
static int maxpool_bn_backward_t(int n, int h, int w, int c, const void* z, const void* dy, const float* stats, void* dz, float* dgamma, float* dbeta,
                                 void* scratch, const BnBackwardExtra& ex, cudaStream_t st) {
    const PoolBn p = pool_windows(n, h, w, c, VEC);
    float* const partial = (float*)scratch;
    float* const coef = partial + (size_t)BN_MAX_BLOCKS * c * 2;
    const unsigned blocks = (unsigned)std::max<int64_t>(1, std::min<int64_t>(pool_blocks(p), POOL_BN_BLOCKS));
    launch(Start::ON_STREAMS, maxpool2x2_bn_sums_kernel<T, VEC>, blocks, 256, 0, st, (const T*)z, (const T*)dy, stats, p, partial);
    CKPT_LAUNCH_CHECK("max-pool 2x2 backward with batch-norm sums");
    launch(Start::ON_STREAMS, bn_finalize_bwd_kernel, (c + FIN_CH - 1) / FIN_CH, FIN_THREADS, 0, st, partial, (int)(2 * blocks), c, 1.0 / (double)(4 * p.windows), stats, dgamma,
           dbeta, coef, ex.gamma, ex.beta);
    CKPT_LAUNCH_CHECK("batch-norm backward finalize");
    launch(Start::ON_STREAMS, maxpool2x2_bn_apply_kernel<T, VEC>, pool_blocks(p), 256, 0, st, (const T*)z,
           (const T*)dy, stats, coef, p, (T*)dz);
    CKPT_LAUNCH_CHECK("max-pool 2x2 backward through batch norm");
    return CKPT_OK;
}
int maxpool_bn_backward(int dtype, int n, int h, int w, int c, const void* z, const void* dy, const float* stats, void* dz, float* dgamma, float* dbeta,
                        void* scratch, void* stream, const BnBackwardExtra& ex) {
    return dtype == CKPT_DTYPE_BF16 ? maxpool_bn_backward_t<__nv_bfloat16, 8>(n, h, w, c, z, dy, stats, dz, dgamma, dbeta, scratch, ex, (cudaStream_t)stream)
                                    : maxpool_bn_backward_t<float, 4>(n, h, w, c, z, dy, stats, dz, dgamma, dbeta, scratch, ex, (cudaStream_t)stream);
}
int maxpool_backward(int dtype, int n, int h, int w, int c, int k, int stride, int pad, const void* x, const void* dy, void* dx, const float* act, void* stream,
                     float* bn_partial, int* bn_blocks, void* scratch, int64_t scratch_bytes) {
    int ho = (h + 2 * pad - k) / stride + 1, wo = (w + 2 * pad - k) / stride + 1;
    if (bn_blocks) *bn_blocks = 0;
    if (pool_2x2(dtype, h, w, c, k, stride, pad)) {
        const int vec = dtype == CKPT_DTYPE_BF16 ? 8 : 4;
        const int64_t items = (int64_t)n * ho * wo * (c / vec);
        if (dtype == CKPT_DTYPE_BF16)
            launch(Start::ON_STREAMS, maxpool2x2_bwd_kernel<__nv_bfloat16, 8>, elementwise_grid(items), 256, 0, (cudaStream_t)stream, (const __nv_bfloat16*)x, (const __nv_bfloat16*)dy, (__nv_bfloat16*)dx, items, wo, ho, c / vec, c, act);
        else
            launch(Start::ON_STREAMS, maxpool2x2_bwd_kernel<float, 4>, elementwise_grid(items), 256, 0, (cudaStream_t)stream, (const float*)x, (const float*)dy, (float*)dx, items, wo, ho, c / vec, c, act);
        CKPT_LAUNCH_CHECK("max-pool 2x2 backward");
        return CKPT_OK;
    }
    if (act && pool_3x3(dtype, c, k, stride, pad)) {
        // batch-norm sums first in the scratch region (the batch-norm backward reads them there), positions behind them
        const int64_t sums = align_up(bn_scratch_bytes(0, c), 256), windows = (int64_t)n * ho * wo * (c / 8);
        if (!scratch || scratch_bytes < sums + windows * 8 || (uintptr_t)scratch % 16) { set_error("pooling scratch too small"); return CKPT_E_WORKSPACE; }
        uint8_t* const arg = (uint8_t*)scratch + sums;
        cudaStream_t st = (cudaStream_t)stream;
        launch(Start::ON_STREAMS, maxpool3_arg_act_kernel, elementwise_grid(windows), 256, 0, st, (const __nv_bfloat16*)x, arg, windows, h, w, c, ho, wo, act);
        CKPT_LAUNCH_CHECK("max-pool 3x3 arg-max");
        const unsigned grid = (unsigned)std::max<int64_t>(1, std::min<int64_t>((windows + 255) / 256, BN_MAX_BLOCKS));
        if (bn_partial && bn_blocks) {
            launch(Start::ON_STREAMS, maxpool3_bwd_kernel<true>, grid, 256, 0, st, arg, (const __nv_bfloat16*)dy, (__nv_bfloat16*)dx, windows, h, w, c, ho, wo, (const __nv_bfloat16*)x, act, bn_partial);
            *bn_blocks = (int)grid;
        } else {
            launch(Start::ON_STREAMS, maxpool3_bwd_kernel<false>, grid, 256, 0, st, arg, (const __nv_bfloat16*)dy, (__nv_bfloat16*)dx, windows, h, w, c, ho, wo, nullptr, nullptr, nullptr);
        }
        CKPT_LAUNCH_CHECK("max-pool backward from arg-max");
        return CKPT_OK;
    }
    if (act) { set_error("the general pooling kernel takes an activated input"); return CKPT_E_BAD_ARG; }
    const int64_t arg_bytes = maxpool_backward_scratch_bytes(dtype, n, h, w, c, k, stride, pad);
    if (arg_bytes > 0 && scratch && scratch_bytes >= arg_bytes && ((uintptr_t)scratch & 7u) == 0) {
        const int vec = dtype == CKPT_DTYPE_BF16 ? 8 : 4;
        const int64_t windows = (int64_t)n * ho * wo * (c / vec), pixels = (int64_t)n * h * w * (c / vec);
        cudaStream_t st = (cudaStream_t)stream;
        if (dtype == CKPT_DTYPE_BF16) {
            launch(Start::ON_STREAMS, maxpool_argmax_kernel<__nv_bfloat16, 8>, elementwise_grid(windows), 256, 0, st, (const __nv_bfloat16*)x, (uint8_t*)scratch, windows, h, w, c, ho, wo, k, stride, pad);
            CKPT_LAUNCH_CHECK("max-pool arg-max");
            if (pool_3x3(dtype, c, k, stride, pad)) launch(Start::ON_STREAMS, maxpool3_bwd_kernel<false>, elementwise_grid(windows), 256, 0, st, (const uint8_t*)scratch, (const __nv_bfloat16*)dy, (__nv_bfloat16*)dx, windows, h, w, c, ho, wo, nullptr, nullptr, nullptr);
            else launch(Start::ON_STREAMS, maxpool_bwd_arg_kernel<__nv_bfloat16, 8>, elementwise_grid(pixels), 256, 0, st, (const uint8_t*)scratch, (const __nv_bfloat16*)dy, (__nv_bfloat16*)dx, pixels, h, w, c, ho, wo, k, stride, pad);
        } else {
            launch(Start::ON_STREAMS, maxpool_argmax_kernel<float, 4>, elementwise_grid(windows), 256, 0, st, (const float*)x, (uint8_t*)scratch, windows, h, w, c, ho, wo, k, stride, pad);
            CKPT_LAUNCH_CHECK("max-pool arg-max");
            launch(Start::ON_STREAMS, maxpool_bwd_arg_kernel<float, 4>, elementwise_grid(pixels), 256, 0, st, (const uint8_t*)scratch, (const float*)dy, (float*)dx, pixels, h, w, c, ho, wo, k, stride, pad);
        }
        CKPT_LAUNCH_CHECK("max-pool backward from arg-max");
        return CKPT_OK;
    }
    if (c % bn_vec(dtype, c) == 0 && bn_vec(dtype, c) > 1) {
        const int64_t items = (int64_t)n * h * w * (c / bn_vec(dtype, c));
        if (dtype == CKPT_DTYPE_BF16)
            launch(Start::ON_STREAMS, maxpool_bwd_vec_kernel<__nv_bfloat16, 8>, elementwise_grid(items), 256, 0, (cudaStream_t)stream, (const __nv_bfloat16*)x, (const __nv_bfloat16*)dy, (__nv_bfloat16*)dx, items, h, w, c, ho, wo, k, stride, pad);
        else
            launch(Start::ON_STREAMS, maxpool_bwd_vec_kernel<float, 4>, elementwise_grid(items), 256, 0, (cudaStream_t)stream, (const float*)x, (const float*)dy, (float*)dx, items, h, w, c, ho, wo, k, stride, pad);
        CKPT_LAUNCH_CHECK("max-pool backward");
        return CKPT_OK;
    }
    unsigned grid = elementwise_grid((int64_t)n * h * w * c);
    if (dtype == CKPT_DTYPE_BF16)
        launch(Start::ON_STREAMS, maxpool_bwd_kernel<__nv_bfloat16>, grid, 256, 0, (cudaStream_t)stream, (const __nv_bfloat16*)x, (const __nv_bfloat16*)dy, (__nv_bfloat16*)dx, n, h, w, c, ho, wo, k, stride, pad);
    else
        launch(Start::ON_STREAMS, maxpool_bwd_kernel<float>, grid, 256, 0, (cudaStream_t)stream, (const float*)x, (const float*)dy, (float*)dx, n, h, w, c, ho, wo, k, stride, pad);
    CKPT_LAUNCH_CHECK("max-pool backward");
    return CKPT_OK;
}

// One block per (image, 32 vectors of channels): eight warps share the positions, four loads in flight each, and their sums
// are added in order.  (A thread per channel walking all positions: 111 us for 32 images of 56 x 56 x 64, 18 now.)
template <typename T, int VEC>
__global__ void __launch_bounds__(256) avgpool_fwd_kernel(const T* x, T* y, int hw, int c) {
    previous_grid_done();
    next_grid_may_start();
    __shared__ float red[8][32][VEC + 1];
    const int lane = threadIdx.x % 32, warp = threadIdx.x / 32, vecs = c / VEC;
    // narrow tensors: the lanes of a warp cover several positions
    const int tiles = (vecs + 31) / 32, img = blockIdx.x / tiles;
    const int width = min(vecs, 32), rows = 32 / width, v = blockIdx.x % tiles * 32 + lane % width, row = lane / width;
    const bool active = v < vecs && row < rows;
    const T* src = x + (size_t)img * hw * c + (size_t)v * VEC;
    float s[VEC];
#pragma unroll
    for (int k = 0; k < VEC; ++k) s[k] = 0.f;
    if (active) {
        const int hop = 8 * rows;
        for (int p = warp * rows + row; p < hw; p += 4 * hop) {
            RawVec<T, VEC> r[4];
#pragma unroll
            for (int u = 0; u < 4; ++u)
                if (p + u * hop < hw) r[u] = load_raw<T, VEC>(src + (size_t)(p + u * hop) * c);
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                if (p + u * hop >= hw) break;
                float f[VEC];
                unpack<T, VEC>(r[u], f);
#pragma unroll
                for (int k = 0; k < VEC; ++k) s[k] += f[k];
            }
        }
    }
#pragma unroll
    for (int k = 0; k < VEC; ++k) red[warp][lane][k] = s[k];
    __syncthreads();
    if (warp == 0 && row == 0 && v < vecs) {
#pragma unroll
        for (int k = 0; k < VEC; ++k) s[k] = 0.f;
        for (int w = 0; w < 8; ++w)
            for (int r = 0; r < rows; ++r)
#pragma unroll
                for (int k = 0; k < VEC; ++k) s[k] += red[w][r * width + lane][k];
#pragma unroll
        for (int k = 0; k < VEC; ++k) s[k] /= (float)hw;
        store_vec<T, VEC>(y + (size_t)img * c + (size_t)v * VEC, s);
    }
}
template <typename T, int VEC>
__global__ void __launch_bounds__(256) avgpool_bwd_kernel(const T* dy, T* dx, int64_t vecs, int hw, int lanes) {
    previous_grid_done();
    next_grid_may_start();
    const float area = (float)hw;
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < vecs; i += (int64_t)gridDim.x * blockDim.x) {
        const int64_t pix = i / lanes;
        float g[VEC];
        load_vec<T, VEC>(dy + ((pix / hw) * lanes + i % lanes) * VEC, g);
#pragma unroll
        for (int k = 0; k < VEC; ++k) g[k] = g[k] / area;
        store_vec<T, VEC>(dx + i * VEC, g);
    }
}
template <typename T, int VEC>
static void launch_avgpool_fwd(int n, int hw, int c, const void* x, void* y, cudaStream_t st) {
    launch(Start::ON_STREAMS, avgpool_fwd_kernel<T, VEC>, (unsigned)n * (unsigned)((c / VEC + 31) / 32), 256, 0, st, (const T*)x, (T*)y, hw, c);
}
template <typename T, int VEC>
static void launch_avgpool_bwd(int n, int hw, int c, const void* dy, void* dx, cudaStream_t st) {
    const int64_t vecs = (int64_t)n * hw * c / VEC;
    launch(Start::ON_STREAMS, avgpool_bwd_kernel<T, VEC>, elementwise_grid(vecs), 256, 0, st, (const T*)dy, (T*)dx, vecs, hw, c / VEC);
}
int avgpool_forward(int dtype, int n, int h, int w, int c, const void* x, void* y, void* stream) {
    cudaStream_t st = (cudaStream_t)stream;
    const int vec = dtype == CKPT_DTYPE_BF16 ? 8 : 4;
    const bool wide = c % vec == 0 && aligned16(x) && aligned16(y);
    if (dtype == CKPT_DTYPE_BF16) wide ? launch_avgpool_fwd<__nv_bfloat16, 8>(n, h * w, c, x, y, st) : launch_avgpool_fwd<__nv_bfloat16, 1>(n, h * w, c, x, y, st);
    else wide ? launch_avgpool_fwd<float, 4>(n, h * w, c, x, y, st) : launch_avgpool_fwd<float, 1>(n, h * w, c, x, y, st);
    CKPT_LAUNCH_CHECK("average-pool forward");
    return CKPT_OK;
}
int avgpool_backward(int dtype, int n, int h, int w, int c, const void* dy, void* dx, void* stream) {
    cudaStream_t st = (cudaStream_t)stream;
    const int vec = dtype == CKPT_DTYPE_BF16 ? 8 : 4;
    const bool wide = c % vec == 0 && aligned16(dy) && aligned16(dx);
    if (dtype == CKPT_DTYPE_BF16) wide ? launch_avgpool_bwd<__nv_bfloat16, 8>(n, h * w, c, dy, dx, st) : launch_avgpool_bwd<__nv_bfloat16, 1>(n, h * w, c, dy, dx, st);
    else wide ? launch_avgpool_bwd<float, 4>(n, h * w, c, dy, dx, st) : launch_avgpool_bwd<float, 1>(n, h * w, c, dy, dx, st);
    CKPT_LAUNCH_CHECK("average-pool backward");
    return CKPT_OK;
}

// ================================================================================================
// Small helpers for the fully connected units and the losses
// ================================================================================================
template <typename T>
__global__ void relu_mask_kernel(T* g, const T* y, int64_t elems) {
    previous_grid_done();
    next_grid_may_start();
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < elems; i += (int64_t)gridDim.x * blockDim.x)
        if (!(ld(y + i) > 0.f)) g[i] = cvt<T>(0.f);
}
// 16-byte form: g is rewritten whole (the kept elements unchanged), four packed loads per operand in flight.
template <typename T, int VEC>
__global__ void __launch_bounds__(256) relu_mask_vec_kernel(T* g, const T* y, int64_t vecs) {
    previous_grid_done();
    next_grid_may_start();
    constexpr int U = 4;
    for (int64_t i0 = (int64_t)blockIdx.x * (256 * U) + threadIdx.x; i0 < vecs; i0 += (int64_t)gridDim.x * (256 * U)) {
        RawVec<T, VEC> rg[U], ry[U];
#pragma unroll
        for (int u = 0; u < U; ++u)
            if (i0 + u * 256 < vecs) { rg[u] = load_raw<T, VEC>(g + (i0 + u * 256) * VEC); ry[u] = load_raw<T, VEC>(y + (i0 + u * 256) * VEC); }
#pragma unroll
        for (int u = 0; u < U; ++u) {
            if (i0 + u * 256 >= vecs) break;
            float gv[VEC], yv[VEC], o[VEC];
            unpack<T, VEC>(rg[u], gv);
            unpack<T, VEC>(ry[u], yv);
#pragma unroll
            for (int k = 0; k < VEC; ++k) o[k] = yv[k] > 0.f ? gv[k] : 0.f;
            store_vec<T, VEC>(g + (i0 + u * 256) * VEC, o);
        }
    }
}
int relu_mask_inplace(int dtype, int64_t elems, void* g, const void* y, void* stream) {
    cudaStream_t st = (cudaStream_t)stream;
    const int vec = dtype == CKPT_DTYPE_BF16 ? 8 : 4;
    if (elems % vec == 0 && aligned16(g) && aligned16(y)) {
        const int64_t vecs = elems / vec;
        const unsigned grid = (unsigned)std::max<int64_t>(1, std::min<int64_t>((vecs + 1023) / 1024, 148 * 32));
        if (dtype == CKPT_DTYPE_BF16) launch(Start::ON_STREAMS, relu_mask_vec_kernel<__nv_bfloat16, 8>, grid, 256, 0, st, (__nv_bfloat16*)g, (const __nv_bfloat16*)y, vecs);
        else launch(Start::ON_STREAMS, relu_mask_vec_kernel<float, 4>, grid, 256, 0, st, (float*)g, (const float*)y, vecs);
    } else if (dtype == CKPT_DTYPE_BF16) {
        launch(Start::ON_STREAMS, relu_mask_kernel<__nv_bfloat16>, elementwise_grid(elems), 256, 0, st, (__nv_bfloat16*)g, (const __nv_bfloat16*)y, elems);
    } else {
        launch(Start::ON_STREAMS, relu_mask_kernel<float>, elementwise_grid(elems), 256, 0, st, (float*)g, (const float*)y, elems);
    }
    CKPT_LAUNCH_CHECK("ReLU mask");
    return CKPT_OK;
}

// ReLU as a chain unit of its own: 16-byte accesses, scalar tail.  y may alias x, dx may alias dy.
template <typename T>
__global__ void __launch_bounds__(256) relu_fwd_kernel(const T* x, T* y, int64_t elems) {
    previous_grid_done();
    next_grid_may_start();
    constexpr int V = 16 / sizeof(T);
    const int64_t vecs = elems / V;
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < vecs; i += (int64_t)gridDim.x * blockDim.x) {
        uint4 raw = reinterpret_cast<const uint4*>(x)[i];
        T* e = reinterpret_cast<T*>(&raw);
#pragma unroll
        for (int k = 0; k < V; ++k) e[k] = cvt<T>(fmaxf(ld(e + k), 0.f));
        reinterpret_cast<uint4*>(y)[i] = raw;
    }
    if (blockIdx.x == 0)
        for (int64_t i = vecs * V + threadIdx.x; i < elems; i += blockDim.x) y[i] = cvt<T>(fmaxf(ld(x + i), 0.f));
}
template <typename T>
__global__ void __launch_bounds__(256) relu_bwd_kernel(const T* dy, const T* y, T* dx,
                                                       int64_t elems) {
    previous_grid_done();
    next_grid_may_start();
    constexpr int V = 16 / sizeof(T);
    const int64_t vecs = elems / V;
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < vecs; i += (int64_t)gridDim.x * blockDim.x) {
        uint4 g = reinterpret_cast<const uint4*>(dy)[i];
        uint4 o = reinterpret_cast<const uint4*>(y)[i];
        T* ge = reinterpret_cast<T*>(&g);
        const T* oe = reinterpret_cast<const T*>(&o);
#pragma unroll
        for (int k = 0; k < V; ++k) if (!(ld(oe + k) > 0.f)) ge[k] = cvt<T>(0.f);
        reinterpret_cast<uint4*>(dx)[i] = g;
    }
    if (blockIdx.x == 0)
        for (int64_t i = vecs * V + threadIdx.x; i < elems; i += blockDim.x) dx[i] = ld(y + i) > 0.f ? dy[i] : cvt<T>(0.f);
}
int relu_forward(int dtype, int64_t elems, const void* x, void* y, void* stream) {
    const int64_t vecs = elems / (dtype == CKPT_DTYPE_BF16 ? 8 : 4);
    if (dtype == CKPT_DTYPE_BF16) launch(Start::ON_STREAMS, relu_fwd_kernel<__nv_bfloat16>, elementwise_grid(vecs), 256, 0, (cudaStream_t)stream, (const __nv_bfloat16*)x, (__nv_bfloat16*)y, elems);
    else launch(Start::ON_STREAMS, relu_fwd_kernel<float>, elementwise_grid(vecs), 256, 0, (cudaStream_t)stream, (const float*)x, (float*)y, elems);
    CKPT_LAUNCH_CHECK("ReLU forward");
    return CKPT_OK;
}
int relu_backward(int dtype, int64_t elems, const void* dy, const void* y, void* dx, void* stream) {
    const int64_t vecs = elems / (dtype == CKPT_DTYPE_BF16 ? 8 : 4);
    if (dtype == CKPT_DTYPE_BF16) launch(Start::ON_STREAMS, relu_bwd_kernel<__nv_bfloat16>, elementwise_grid(vecs), 256, 0, (cudaStream_t)stream, (const __nv_bfloat16*)dy, (const __nv_bfloat16*)y, (__nv_bfloat16*)dx, elems);
    else launch(Start::ON_STREAMS, relu_bwd_kernel<float>, elementwise_grid(vecs), 256, 0, (cudaStream_t)stream, (const float*)dy, (const float*)y, (float*)dx, elems);
    CKPT_LAUNCH_CHECK("ReLU backward");
    return CKPT_OK;
}

// A block sums 32 columns, eight threads each.
template <typename T>
__global__ void __launch_bounds__(256) column_sum_kernel(const T* g, float* out, int64_t rows, int c, SgdUpdate upd) {
    previous_grid_done();
    next_grid_may_start();
    __shared__ float red[8][32];
    const int lane = threadIdx.x % 32, part = threadIdx.x / 32, ch = blockIdx.x * 32 + lane;
    float s = 0.f;
    if (ch < c) {
#pragma unroll 4
        for (int64_t r = part; r < rows; r += 8) s += ld(g + r * c + ch);
    }
    red[part][lane] = s;
    __syncthreads();
    if (part != 0 || ch >= c) return;
    for (int q = 1; q < 8; ++q) s += red[q][lane];
    out[ch] = s;
    if (upd.w) { float* w = (float*)upd.w + ch; *w = fmaf(-upd.lr, s, *w); }
}
int column_sums(int dtype, int64_t rows, int c, const void* g, float* out, void* stream, const SgdUpdate& upd) {
    if (dtype == CKPT_DTYPE_BF16) launch(Start::ON_STREAMS, column_sum_kernel<__nv_bfloat16>, (c + 31) / 32, 256, 0, (cudaStream_t)stream, (const __nv_bfloat16*)g, out, rows, c, upd);
    else launch(Start::ON_STREAMS, column_sum_kernel<float>, (c + 31) / 32, 256, 0, (cudaStream_t)stream, (const float*)g, out, rows, c, upd);
    CKPT_LAUNCH_CHECK("column sums");
    return CKPT_OK;
}

// One block per sample: max, sum of exponentials, loss term, gradient (softmax - onehot)/batch.
template <typename T>
__global__ void __launch_bounds__(256) softmax_ce_kernel(const T* logits, const int32_t* labels,
                                                         int classes, float inv_batch, float* row_loss,
                                                         T* dlogits) {
    previous_grid_done();
    next_grid_may_start();
    __shared__ float red[256];
    const T* row = logits + (size_t)blockIdx.x * classes;
    float m = -INFINITY;
    for (int i = threadIdx.x; i < classes; i += 256) m = fmaxf(m, ld(row + i));
    red[threadIdx.x] = m;
    __syncthreads();
    for (int s = 128; s > 0; s >>= 1) { if (threadIdx.x < s) red[threadIdx.x] = fmaxf(red[threadIdx.x], red[threadIdx.x + s]); __syncthreads(); }
    m = red[0];
    __syncthreads();
    float sum = 0.f;
    for (int i = threadIdx.x; i < classes; i += 256) sum += expf(ld(row + i) - m);
    red[threadIdx.x] = sum;
    __syncthreads();
    for (int s = 128; s > 0; s >>= 1) { if (threadIdx.x < s) red[threadIdx.x] += red[threadIdx.x + s]; __syncthreads(); }
    sum = red[0];
    const int label = labels[blockIdx.x];
    const float inv_sum = 1.f / sum;
    for (int i = threadIdx.x; i < classes; i += 256) {
        float p = expf(ld(row + i) - m) * inv_sum;
        dlogits[(size_t)blockIdx.x * classes + i] = cvt<T>((p - (i == label ? 1.f : 0.f)) * inv_batch);
    }
    if (threadIdx.x == 0) row_loss[blockIdx.x] = logf(sum) + m - ld(row + label);
}
__global__ void mean_rows_kernel(const float* row_loss, int batch, float* loss) {
    previous_grid_done();
    next_grid_may_start();
    if (threadIdx.x == 0 && blockIdx.x == 0) {
        double s = 0.0;
        for (int i = 0; i < batch; ++i) s += row_loss[i];
        *loss = (float)(s / batch);
    }
}
int softmax_ce(int dtype, int batch, int classes, const void* logits, const int32_t* labels, float* loss, void* dlogits,
               float* row_scratch, void* stream) {
    cudaStream_t st = (cudaStream_t)stream;
    if (dtype == CKPT_DTYPE_BF16)
        launch(Start::ON_STREAMS, softmax_ce_kernel<__nv_bfloat16>, batch, 256, 0, st, (const __nv_bfloat16*)logits, labels, classes, 1.f / batch, row_scratch, (__nv_bfloat16*)dlogits);
    else
        launch(Start::ON_STREAMS, softmax_ce_kernel<float>, batch, 256, 0, st, (const float*)logits, labels, classes, 1.f / batch, row_scratch, (float*)dlogits);
    CKPT_LAUNCH_CHECK("softmax cross-entropy");
    launch(Start::ON_STREAMS, mean_rows_kernel, 1, 32, 0, st, row_scratch, batch, loss);
    CKPT_LAUNCH_CHECK("loss mean");
    return CKPT_OK;
}

constexpr int SUM_BLOCKS = 256;
template <typename T>
__global__ void __launch_bounds__(256) sum_partial_kernel(const T* y, int64_t elems, double* partial,
                                                          T* grad) {
    previous_grid_done();
    next_grid_may_start();
    __shared__ double red[256];
    double s = 0.0;
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < elems; i += (int64_t)gridDim.x * blockDim.x) {
        s += (double)ld(y + i);
        grad[i] = cvt<T>(1.f);
    }
    red[threadIdx.x] = s;
    __syncthreads();
    for (int k = 128; k > 0; k >>= 1) { if (threadIdx.x < k) red[threadIdx.x] += red[threadIdx.x + k]; __syncthreads(); }
    if (threadIdx.x == 0) partial[blockIdx.x] = red[0];
}
__global__ void sum_final_kernel(const double* partial, int blocks, double* loss) {
    previous_grid_done();
    next_grid_may_start();
    if (threadIdx.x == 0 && blockIdx.x == 0) {
        double s = 0.0;
        for (int i = 0; i < blocks; ++i) s += partial[i];
        *loss = s;
    }
}
int64_t sum_loss_scratch_bytes() { return SUM_BLOCKS * (int64_t)sizeof(double); }
int sum_loss(int dtype, int64_t elems, const void* y, double* loss, void* grad, double* scratch, void* stream) {
    cudaStream_t st = (cudaStream_t)stream;
    if (dtype == CKPT_DTYPE_BF16) launch(Start::ON_STREAMS, sum_partial_kernel<__nv_bfloat16>, SUM_BLOCKS, 256, 0, st, (const __nv_bfloat16*)y, elems, scratch, (__nv_bfloat16*)grad);
    else launch(Start::ON_STREAMS, sum_partial_kernel<float>, SUM_BLOCKS, 256, 0, st, (const float*)y, elems, scratch, (float*)grad);
    CKPT_LAUNCH_CHECK("sum loss");
    launch(Start::ON_STREAMS, sum_final_kernel, 1, 32, 0, st, scratch, SUM_BLOCKS, loss);
    CKPT_LAUNCH_CHECK("sum loss final");
    return CKPT_OK;
}

__global__ void copy_kernel(uint4* dst, const uint4* src, int64_t vecs) {
    previous_grid_done();
    next_grid_may_start();
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < vecs; i += (int64_t)gridDim.x * blockDim.x) dst[i] = src[i];
}
int device_copy(void* dst, const void* src, int64_t bytes, void* stream) {
    // sizes and offsets inside the arena and the workspace are multiples of 256 bytes
    int64_t vecs = bytes / 16;
    launch(Start::ON_STREAMS, copy_kernel, elementwise_grid(vecs), 256, 0, (cudaStream_t)stream, (uint4*)dst, (const uint4*)src, vecs);
    CKPT_LAUNCH_CHECK("gradient carry copy");
    return CKPT_OK;
}

// w <- w - lr * g, element by element (float32 arithmetic; bf16 parameters rounded to nearest even).
template <typename T>
__global__ void sgd_update_kernel(T* w, const float* g, int64_t elems, float lr) {
    previous_grid_done();
    next_grid_may_start();
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < elems; i += (int64_t)gridDim.x * blockDim.x) {
        if constexpr (sizeof(T) == 2) w[i] = __float2bfloat16_rn(fmaf(-lr, g[i], __bfloat162float(w[i])));
        else w[i] = fmaf(-lr, g[i], w[i]);
    }
}
int sgd_update(const SgdUpdate& u, const float* g, int64_t elems, void* stream) {
    if (!u.w || elems <= 0) return CKPT_OK;
    if (u.dtype == CKPT_DTYPE_BF16) launch(Start::ON_STREAMS, sgd_update_kernel<__nv_bfloat16>, elementwise_grid(elems), 256, 0, (cudaStream_t)stream, (__nv_bfloat16*)u.w, g, elems, u.lr);
    else launch(Start::ON_STREAMS, sgd_update_kernel<float>, elementwise_grid(elems), 256, 0, (cudaStream_t)stream, (float*)u.w, g, elems, u.lr);
    CKPT_LAUNCH_CHECK("parameter update");
    return CKPT_OK;
}

}  // namespace ckpt
