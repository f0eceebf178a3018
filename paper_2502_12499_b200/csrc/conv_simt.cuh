// CUDA-core implicit-GEMM convolution: C[M][N] = sum_k A(m,k) * B(k,n), any filter size, stride, padding and channel
// count, float32 or bfloat16 storage, float32 FMA arithmetic.
//   MODE 0 forward: M = pixels out, N = c_out,     K = k*k*c_in      A gathered from x (K contiguous), B = w (K contiguous)
//   MODE 1 dgrad  : M = pixels in,  N = c_in,      K = k*k*c_out     A gathered from dz (K contiguous), B = w (N contiguous)
//   MODE 2 wgrad  : M = c_out,      N = k*k*c_in,  K = pixels out    A = dz (M contiguous), B gathered from x (N contiguous)
//
// Bound: FMA issue on large shapes, latency on small ones (the layers of a 32 x 32 image leave most SMs without a tile).
// Operand tiles go to shared memory as they lie in memory, 64 bytes of K per row (or that many K rows), by 16-byte
// asynchronous copies, STAGES deep, so the copies of the next stages run under the FMAs of this one and a short
// reduction is in flight as a whole; a thread keeps a TM x TN block and reads its operands 16 bytes at a time.  The
// reduction of a tile can be split over the CTAs of a cluster, whose partial tiles are added over distributed shared
// memory in rank order (one launch, no scratch), and a weight gradient's over further slices whose partial sums another
// kernel adds in slice order.  Every summation order is fixed by the shape.
// A sum is taken in chains of kChain products, whose totals are added: a chain of 1152 has two to three times the error.
// Measured (float32, forward / dgrad / wgrad in us, replayed; in brackets one chain per sum, whose registers let an SM hold more
// CTAs): 32 x 16 x 16 x 64 -> 64 3x3 29/30/22 (27/28/27); 32 x 8 x 8 x 128 -> 128 29/28/22 (51/52/36); 16 x 112 x 112 x 64 -> 64
// 405/424/353 (431/438/453; 37 of the 72 TFLOP/s of the FMA units); 16 x 28 x 28 x 256 -> 256 3x3 stride 2 125/206/100 (165/320/148);
// 4 x 32 x 32 x 16 -> 16 8/8/8 (8/9/9).  At equal plans the chains cost 2-4 %, 128-wide weight-gradient tiles 7 %.  What stands
// between is the issue of everything but FMAs - shared-memory reads, addresses and bounds of the copies - and their latency at 16
// warps per SM.
#pragma once
#include <cooperative_groups.h>
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include <algorithm>
#include <cstdint>

#include "internal.h"
#include "overlap.cuh"

namespace ckpt {
namespace simt {

constexpr int kStages = 4;
constexpr int kChain = 64;         // additions in a row (see the kernel)
enum class Form { CHAINS, WIDE, ONE_CHAIN };

template <typename T> __device__ __forceinline__ float to_f(T v);
template <> __device__ __forceinline__ float to_f<float>(float v) { return v; }
template <> __device__ __forceinline__ float to_f<__nv_bfloat16>(__nv_bfloat16 v) { return __bfloat162float(v); }
template <typename T> __device__ __forceinline__ T from_f(float v);
template <> __device__ __forceinline__ float from_f<float>(float v) { return v; }
template <> __device__ __forceinline__ __nv_bfloat16 from_f<__nv_bfloat16>(float v) { return __float2bfloat16_rn(v); }

// N (2 or 4) consecutive values of a shared-memory row
template <typename T, int N>
__device__ __forceinline__ void lds(const T* p, float* v) {
    if constexpr (sizeof(T) == 4) {
        if constexpr (N == 4) {
            const float4 t = *reinterpret_cast<const float4*>(p);
            v[0] = t.x; v[1] = t.y; v[2] = t.z; v[3] = t.w;
        } else {
            const float2 t = *reinterpret_cast<const float2*>(p);
            v[0] = t.x; v[1] = t.y;
        }
    } else {
        uint32_t w[N / 2];
        if constexpr (N == 4) { const uint2 t = *reinterpret_cast<const uint2*>(p); w[0] = t.x; w[1] = t.y; }
        else w[0] = *reinterpret_cast<const uint32_t*>(p);
#pragma unroll
        for (int i = 0; i < N / 2; ++i) { v[2 * i] = __uint_as_float(w[i] << 16); v[2 * i + 1] = __uint_as_float(w[i] & 0xffff0000u); }
    }
}

__device__ __forceinline__ void copy16(void* dst, const void* src, bool in) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"((uint32_t)__cvta_generic_to_shared(dst)), "l"(src), "r"(in ? 16 : 0) : "memory");
}
__device__ __forceinline__ void copy4(void* dst, const void* src, bool in) {
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;" ::"r"((uint32_t)__cvta_generic_to_shared(dst)), "l"(src), "r"(in ? 4 : 0) : "memory");
}

template <typename T, int MODE, int BM, int BN, int TM, int TN>
struct Tile {
    static constexpr int threads = (BM / TM) * (BN / TN);
    static constexpr int V = 16 / (int)sizeof(T);            // values of a 16-byte chunk
    static constexpr int BK = 4 * V;                         // reduction depth of a stage
    static constexpr bool a_k = MODE != 2, b_k = MODE == 0;  // K contiguous in shared memory (and in memory)
    // row lengths in values; one chunk of padding puts consecutive rows on different banks
    static constexpr int a_row = a_k ? BK + V : BM + V, b_row = b_k ? BK + V : BN + V;
    static constexpr int a_rows = a_k ? BM : BK, b_rows = b_k ? BN : BK;
    static constexpr int a_elems = a_rows * a_row, b_elems = b_rows * b_row;
    static constexpr int stage_bytes = (a_elems + b_elems) * (int)sizeof(T);
    static constexpr int smem = kStages * stage_bytes > BM * BN * 4 ? kStages * stage_bytes : BM * BN * 4;
    // CTAs that an SM shall hold - what the kernel is compiled for and what the plan counts on: by the registers for the chain and
    // the total of a block, operands and addresses, and by shared memory
    static constexpr int by_registers = TM * TN >= 64 ? 256 / threads : TM * TN >= 32 ? (sizeof(T) == 4 ? 4 : 3) : TM * TN >= 16 ? 5 : 7;
    static constexpr int by_memory = 228 * 1024 / (smem + 1024);
    static constexpr int held = by_registers < by_memory ? by_registers : by_memory;
    static constexpr int held_values = MODE == 2 && TM * TN >= 32 && held < 4 ? 4 : held;      // operands fetched value by value (shapes 2, 4 and 6)
    static constexpr int held_one = TM * TN >= 32 ? (sizeof(T) == 4 ? 5 : 4) : TM * TN >= 16 ? (sizeof(T) == 4 ? 6 : 5) : 8;      // a chain at most
};

// A position along K of modes 0 and 1: channel within a filter position, and the filter position as (row, column) indices.
struct TapPos {
    int c, r, s;
    __device__ __forceinline__ void set(int kk, int channels, int cols) { const int t = kk / channels; c = kk % channels; r = t / cols; s = t % cols; }
    __device__ __forceinline__ void advance(int by, int channels, int cols) {
        c += by;
        while (c >= channels) { c -= channels; if (++s == cols) { s = 0; ++r; } }
    }
};
// A pixel of an n x H x W grid, walked in steps
struct Pixel {
    int w, h, n;
    __device__ __forceinline__ void set(int p, int W, int H) { w = p % W; const int t = p / W; h = t % H; n = t / H; }
    __device__ __forceinline__ void advance(int by, int W, int H) {
        w += by;
        while (w >= W) { w -= W; if (++h == H) { h = 0; ++n; } }
    }
};

// VA / VB: the operand is fetched in 16-byte chunks (its contiguous dimension is a multiple of a chunk and 16-byte
// aligned); otherwise value by value: float32 by asynchronous copies too, bfloat16 through registers, loaded before the FMAs
// of a step and stored after them.  A forward layer of that kind often has a short reduction (27 values for three input
// channels), whose last step stops where it ends (3 -> 256, 1x1, 49 images of 78 x 18, bfloat16: 81 us with whole steps, 46).
// sums (mode 0, or null): batch-norm sums of the stored values, a row pair [sum | sum of squares][N] per CTA that stores a share of
// a tile (a pass of its own costs its launch and 2.4-4.6 us: eight units of 16 channels, 4 images of 32 x 32, launched one by one 400 -> 379 us,
// a float32 VGG-16 on 32 images 1154 -> 1131).
// gridDim.z = slices * cluster; slice z of the reduction starts at z * k_per_slice (a multiple of BK).
// Mode 1 with a stride: the input pixels fall into stride x stride parity classes, each reached by every stride-th filter
// row and column only; a block works on one class (classes follow one another in blockIdx.x) and its K covers just those.
// FORM (modes 0, 1): WIDE, chunks of A through filters of more than 16 rows, whose places outside the tensor are found by coordinates;
// ONE_CHAIN, value by value, a reduction of one chain at most per CTA, without the registers of a second set of sums (us, with
// them -> so: 3 -> 64 3x3 at 224 x 224, 16 images, float32 166 -> 147, 3 -> 64 1x1 at 40 x 40, 20 images, bfloat16 11.9 -> 7.8).
template <typename T, int MODE, int BM, int BN, int TM, int TN, bool VA, bool VB, Form FORM>
__global__ void __launch_bounds__((BM / TM) * (BN / TN), (FORM == Form::ONE_CHAIN ? Tile<T, MODE, BM, BN, TM, TN>::held_one : VA && VB ? Tile<T, MODE, BM, BN, TM, TN>::held : Tile<T, MODE, BM, BN, TM, TN>::held_values))
conv_gemm_kernel(ConvGeom g, const T* A, const T* B, void* out, const float* bias,
                 int relu, int M, int N, int K, int k_per_slice, int cluster, SgdUpdate upd, float* sums) {
    previous_grid_done();
    next_grid_may_start();
    using L = Tile<T, MODE, BM, BN, TM, TN>;
    constexpr int NT = L::threads, V = L::V, BK = L::BK;
    constexpr bool WIDE = FORM == Form::WIDE, ONE = FORM == Form::ONE_CHAIN;
    extern __shared__ __align__(16) uint8_t smem[];
    T* const stages = reinterpret_cast<T*>(smem);
    const int tid = threadIdx.x;
    const int n0 = blockIdx.y * BN;
    // mode 1: parity class of this block and its filter rows r0, r0 + stride, .. (rows of them; likewise columns)
    int bx = blockIdx.x, ph = 0, pw = 0, r0 = 0, s0 = 0, cols = g.k, W = MODE == 0 ? g.wo : g.w, H = MODE == 0 ? g.ho : g.h;
    if (MODE == 1 && g.stride > 1) {
        const int per_class = gridDim.x / (g.stride * g.stride);
        ph = bx / per_class / g.stride; pw = bx / per_class % g.stride; bx %= per_class;
        r0 = (ph + g.pad) % g.stride; s0 = (pw + g.pad) % g.stride;
        const int rows = r0 < g.k ? (g.k - r0 - 1) / g.stride + 1 : 0;
        cols = s0 < g.k ? (g.k - s0 - 1) / g.stride + 1 : 0;
        H = (g.h - ph + g.stride - 1) / g.stride; W = (g.w - pw + g.stride - 1) / g.stride;
        M = g.n * H * W; K = rows * cols * g.cout;
        if (K == 0) cols = 1;
    }
    const int m0 = bx * BM;
    if (m0 >= M) return;                                      // a class smaller than the largest (the whole cluster leaves)
    const int k_begin = min(K, (int)blockIdx.z * k_per_slice), k_end = min(K, k_begin + k_per_slice);
    const int steps = (k_end - k_begin + BK - 1) / BK;
    const int kc = MODE == 0 ? g.cin : g.cout;               // channels per filter position along K (modes 0, 1)

    // address of A at pixel (ih / th base, iw / tw base) of image n for a filter position, or null outside the tensor
    auto a_ptr = [&](int n, int bh, int bw, const TapPos& t) -> const T* {
        if (MODE == 0) {
            const int ih = bh + t.r, iw = bw + t.s;
            if ((unsigned)ih >= (unsigned)g.h || (unsigned)iw >= (unsigned)g.w) return nullptr;
            return A + (int64_t)(((uint32_t)n * g.h + ih) * g.w + iw) * g.cin + t.c;
        }
        const int th = bh - t.r, tw = bw - t.s;
        if ((unsigned)th >= (unsigned)g.ho || (unsigned)tw >= (unsigned)g.wo) return nullptr;
        return A + (int64_t)(((uint32_t)n * g.ho + th) * g.wo + tw) * g.cout + t.c;
    };
    // corner of a pixel's window in the gathered tensor.  Mode 1: output row of filter row r0 + stride * t is base - t
    auto a_base_h = [&](int h) { return MODE == 0 ? h * g.stride - g.pad : (h * g.stride + ph + g.pad - r0) / g.stride; };
    auto a_base_w = [&](int w) { return MODE == 0 ? w * g.stride - g.pad : (w * g.stride + pw + g.pad - s0) / g.stride; };
    // value (tap position, n) of the filter in mode 1
    auto b_off = [&](const TapPos& t) { return (int64_t)(((uint32_t)t.c * g.k + r0 + t.r * g.stride) * g.k + s0 + t.s * g.stride) * g.cin; };

    // ---- what a thread fetches in every stage: chunk c = tid + i * NT of each tile, or value e = tid + i * NT
    constexpr int a_len = (VA ? 1 : V) * (L::a_k ? 4 : BM / V), b_len = (VB ? 1 : V) * (L::b_k ? 4 : BN / V);      // items of a row
    constexpr int a_items = L::a_rows * a_len, b_items = L::b_rows * b_len;
    constexpr int CA = (a_items + NT - 1) / NT, CB = (b_items + NT - 1) / NT;
    static_assert(NT % a_len == 0 && NT % b_len == 0, "a thread keeps its place in a row");
    constexpr int a_dr = NT / a_len, b_dr = NT / b_len, a_w = VA ? V : 1, b_w = VB ? V : 1;                          // rows apart, values
    const int a_c = tid % a_len * a_w, a_r = tid / a_len, b_c = tid % b_len * b_w, b_r = tid / b_len;
    TapPos a_pos = {0, 0, 0};                                 // modes 0, 1: this thread's place along K
    // chunks: the corner of a row's window, and which filter rows (low half) and columns (high half) of it lie inside the
    // tensor (up to 16 of each): an address is one addition per step, and no multiplication
    const T* a_corner[VA ? CA : 1];
    uint32_t a_inside[VA ? CA : 1];
    int a_top[WIDE ? CA : 1], a_left[WIDE ? CA : 1];          // WIDE: the corner's place
    if (MODE != 2) {
        a_pos.set(k_begin + a_c, kc, cols);
        if (VA) {
#pragma unroll
            for (int i = 0; i < CA; ++i) {
                const int m = m0 + a_r + i * a_dr;
                Pixel p;
                p.set(min(m, M - 1), W, H);
                const int bh = a_base_h(p.h), bw = a_base_w(p.w), th = MODE == 0 ? g.h : g.ho, tw = MODE == 0 ? g.w : g.wo;
                a_corner[VA ? i : 0] = A + (((int64_t)p.n * th + bh) * tw + bw) * kc;
                if (WIDE) { a_top[WIDE ? i : 0] = m < M ? bh : -(1 << 28); a_left[WIDE ? i : 0] = bw; continue; }
                uint32_t inside = 0u;
                for (int t = 0; t < g.k && m < M; ++t) {
                    const int ih = MODE == 0 ? bh + t : bh - t, iw = MODE == 0 ? bw + t : bw - t;
                    inside |= ((unsigned)ih < (unsigned)th ? 1u : 0u) << t | ((unsigned)iw < (unsigned)tw ? 0x10000u : 0u) << t;
                }
                a_inside[VA ? i : 0] = inside;
            }
        }
    }
    TapPos b_pos[VB && MODE == 1 ? CB : 1];                   // mode 1: the rows' places along K
    Pixel b_px[VB && MODE == 2 ? CB : 1];                     // mode 2: the rows' pixels
    int b_tap_h = 0, b_tap_w = 0, b_ci = 0;                   // mode 2: this thread's column
    if (MODE == 1) {
#pragma unroll
        for (int i = 0; i < (VB ? CB : 1); ++i) b_pos[VB && MODE == 1 ? i : 0].set(k_begin + b_r + i * b_dr, g.cout, cols);
    }
    if (MODE == 2) {
        const int n = n0 + b_c, tap = n / g.cin;
        b_ci = n % g.cin; b_tap_w = tap % g.k - g.pad;
        b_tap_h = n < N ? tap / g.k - g.pad : -(1 << 28);
#pragma unroll
        for (int i = 0; i < (VB ? CB : 1); ++i) b_px[VB && MODE == 2 ? i : 0].set(k_begin + b_r + i * b_dr, g.wo, g.ho);
    }
    auto x_ptr = [&](const Pixel& p) -> const T* {            // mode 2: x at this thread's column for an output pixel
        const int ih = p.h * g.stride + b_tap_h, iw = p.w * g.stride + b_tap_w;
        if ((unsigned)ih >= (unsigned)g.h || (unsigned)iw >= (unsigned)g.w) return nullptr;
        return B + (int64_t)(((uint32_t)p.n * g.h + ih) * g.w + iw) * g.cin + b_ci;
    };
    // values fetched through registers (also the filter of an input gradient to a few channels, whose rows of three values are
    // copied no faster: 256 -> 3, 28 images of 13 x 49, float32 85.6 us, 90.6 by copies)
    constexpr bool a_regs = !VA && sizeof(T) == 2, b_regs = !VB && (sizeof(T) == 2 || (MODE == 1 && VA));
    T a_reg[a_regs ? CA : 1], b_reg[b_regs ? CB : 1];

    auto fetch = [&](int step) {
        T* const as_ = stages + (size_t)(step % kStages) * (L::a_elems + L::b_elems);
        T* const bs_ = as_ + L::a_elems;
        const int k0 = k_begin + step * BK;
        Pixel row_px;
        if (!VA && MODE != 2) row_px.set(min(m0 + a_r, M - 1), W, H);
        int64_t a_off = 0;
        uint32_t a_bits = 0u;
        if (VA && MODE != 2 && k0 + a_c < k_end) {
            const int at = a_pos.r * (MODE == 0 ? g.w : g.wo) + a_pos.s;
            a_off = (int64_t)(MODE == 0 ? at : -at) * kc + a_pos.c;
            a_bits = WIDE ? 1u : 1u << a_pos.r | 0x10000u << a_pos.s;
        }
#pragma unroll
        for (int i = 0; i < CA; ++i) {
            const int row = a_r + i * a_dr;
            if (a_items % NT != 0 && row >= L::a_rows) break;
            const T* src = nullptr;
            if (MODE == 2) {
                if (k0 + row < k_end && m0 + a_c < M) src = A + (int64_t)(k0 + row) * g.cout + m0 + a_c;
            } else if (VA) {
                bool in = a_bits != 0u;
                if (WIDE) {
                    const int h = a_top[WIDE ? i : 0], w = a_left[WIDE ? i : 0], ih = MODE == 0 ? h + a_pos.r : h - a_pos.r, iw = MODE == 0 ? w + a_pos.s : w - a_pos.s;
                    in = in && (unsigned)ih < (unsigned)(MODE == 0 ? g.h : g.ho) && (unsigned)iw < (unsigned)(MODE == 0 ? g.w : g.wo);
                } else {
                    in = in && (a_inside[VA ? i : 0] & a_bits) == a_bits;
                }
                if (in) src = a_corner[VA ? i : 0] + a_off;
            } else {
                if (k0 + a_c < k_end && m0 + row < M) src = a_ptr(row_px.n, a_base_h(row_px.h), a_base_w(row_px.w), a_pos);
                row_px.advance(a_dr, W, H);
            }
            if constexpr (VA) copy16(as_ + row * L::a_row + a_c, src ? src : A, src != nullptr);
            else if constexpr (!a_regs) copy4(as_ + row * L::a_row + a_c, src ? src : A, src != nullptr);
            else a_reg[i] = src ? *src : from_f<T>(0.f);
        }
        if (MODE != 2) a_pos.advance(BK, kc, cols);
#pragma unroll
        for (int i = 0; i < CB; ++i) {
            const int row = b_r + i * b_dr;
            if (b_items % NT != 0 && row >= L::b_rows) break;
            const T* src = nullptr;
            if (MODE == 0) {
                if (n0 + row < N && k0 + b_c < k_end) src = B + (int64_t)(n0 + row) * K + k0 + b_c;
            } else {
                const bool in = k0 + row < k_end && n0 + b_c < N;
                constexpr int P = VB ? 1 : 0;
                if (MODE == 1) {
                    TapPos& t = b_pos[MODE == 1 ? P * i : 0];
                    if (in) src = B + b_off(t) + n0 + b_c;
                    t.advance(VB ? BK : b_dr, g.cout, cols);
                } else {
                    Pixel& p = b_px[MODE == 2 ? P * i : 0];
                    if (in) src = x_ptr(p);
                    p.advance(VB ? BK : b_dr, g.wo, g.ho);
                }
            }
            if constexpr (VB) copy16(bs_ + row * L::b_row + b_c, src ? src : B, src != nullptr);
            else if constexpr (!b_regs) copy4(bs_ + row * L::b_row + b_c, src ? src : B, src != nullptr);
            else b_reg[i] = src ? *src : from_f<T>(0.f);
        }
    };
    auto settle = [&](int step) {                             // values fetched through registers
        T* const as_ = stages + (size_t)(step % kStages) * (L::a_elems + L::b_elems);
        T* const bs_ = as_ + L::a_elems;
        if constexpr (a_regs) {
#pragma unroll
            for (int i = 0; i < CA; ++i) {
                const int row = a_r + i * a_dr;
                if (a_items % NT == 0 || row < L::a_rows) as_[row * L::a_row + a_c] = a_reg[i];
            }
        }
        if constexpr (b_regs) {
#pragma unroll
            for (int i = 0; i < CB; ++i) {
                const int row = b_r + i * b_dr;
                if (b_items % NT == 0 || row < L::b_rows) bs_[row * L::b_row + b_c] = b_reg[i];
            }
        }
    };

    // ---- the thread's block: rows and columns are spread so that a warp's reads fall on different banks
    constexpr int TX = BN / TN, TY = BM / TM;
    const int tx = tid % TX, ty = tid / TX;
    constexpr int GM = TM < 4 ? TM : 4, GN = TN < 4 ? TN : 4;         // values per read of an MN-contiguous operand
    auto m_of = [&](int i) { return L::a_k ? ty + i * TY : (i / GM) * (TY * GM) + ty * GM + i % GM; };
    auto n_of = [&](int j) { return L::b_k ? tx + j * TX : (j / GN) * (TX * GN) + tx * GN + j % GN; };
    // chains of kChain products, added up: the error of one float32 chain grows with the square root of its length (in 1e-7 of
    // the result's norm, a chain for the whole reduction -> this: 128 -> 128 3x3 at 28 x 28 6.0 -> 1.6, 512 -> 512 4.3 -> 1.7)
    float acc[TM][TN], total[ONE ? 1 : TM][ONE ? 1 : TN];
#pragma unroll
    for (int i = 0; i < TM; ++i)
#pragma unroll
        for (int j = 0; j < TN; ++j) acc[i][j] = total[ONE ? 0 : i][ONE ? 0 : j] = 0.f;
    auto close_chain = [&] {
        if constexpr (!ONE) {
#pragma unroll
            for (int i = 0; i < TM; ++i)
#pragma unroll
                for (int j = 0; j < TN; ++j) { total[i][j] += acc[i][j]; acc[i][j] = 0.f; }
        }
    };
    auto sum_of = [&](int i, int j) { return ONE ? acc[i][j] : total[ONE ? 0 : i][ONE ? 0 : j]; };

#pragma unroll 1
    for (int p = 0; p < kStages - 1; ++p) {
        if (p < steps) { fetch(p); settle(p); }
        asm volatile("cp.async.commit_group;" ::: "memory");
    }
#pragma unroll 1
    for (int step = 0; step < steps; ++step) {
        asm volatile("cp.async.wait_group %0;" ::"n"(kStages - 2) : "memory");
        __syncthreads();                                      // the stage has landed for all; the one refilled now has been read by all
        const bool more = step + kStages - 1 < steps;
        if (more) fetch(step + kStages - 1);
        asm volatile("cp.async.commit_group;" ::: "memory");
        const T* const as_ = stages + (size_t)(step % kStages) * (L::a_elems + L::b_elems);
        const T* const bs_ = as_ + L::a_elems;
        // Whole steps unrolled, so that shared-memory reads run ahead of the FMAs (float32, at equal plans, us: 3x3 64 -> 64 at 112 x 112,
        // 16 images, forward / input gradient 418/438 with groups of four one at a time, 405/423 so).  Eight by eight blocks and values
        // fetched through registers have none left for more than four groups, 128 x 32 tiles of float32 outputs spill.  In mode 2 the fragments of one k at a time:
        // 64 x 64 tiles 3 % faster than with four fetched in front.
#pragma unroll (TM * TN >= 64 || !(VA && VB) ? 4 : sizeof(T) == 4 && MODE == 0 && BM == 4 * BN ? 1 : BK / 4)
        for (int k4 = 0; k4 < BK; k4 += 4) {
            if (MODE == 0 && !VA && k_begin + step * BK + k4 >= k_end) break;
            float a[TM][L::a_k ? 4 : 1];
            if constexpr (L::a_k) {
#pragma unroll
                for (int i = 0; i < TM; ++i) lds<T, 4>(as_ + m_of(i) * L::a_row + k4, a[i]);
            }
            if constexpr (L::b_k) {
#pragma unroll
                for (int j = 0; j < TN; ++j) {
                    float b[4];
                    lds<T, 4>(bs_ + n_of(j) * L::b_row + k4, b);
#pragma unroll
                    for (int kk = 0; kk < 4; ++kk)
#pragma unroll
                        for (int i = 0; i < TM; ++i) acc[i][j] = fmaf(a[i][kk], b[kk], acc[i][j]);
                }
            } else {
#pragma unroll
                for (int kk = 0; kk < 4; ++kk) {
                    float b[TN];
#pragma unroll
                    for (int j = 0; j < TN; j += GN) lds<T, GN>(bs_ + (k4 + kk) * L::b_row + n_of(j), b + j);
                    if constexpr (!L::a_k) {
#pragma unroll
                        for (int i = 0; i < TM; i += GM) {
                            float t[GM];
                            lds<T, GM>(as_ + (k4 + kk) * L::a_row + m_of(i), t);
#pragma unroll
                            for (int e = 0; e < GM; ++e) a[i + e][0] = t[e];
                        }
                    }
#pragma unroll
                    for (int i = 0; i < TM; ++i)
#pragma unroll
                        for (int j = 0; j < TN; ++j) acc[i][j] = fmaf(a[i][L::a_k ? kk : 0], b[j], acc[i][j]);
                }
            }
        }
        if (more) settle(step + kStages - 1);
        if (step % (kChain / BK) == kChain / BK - 1) close_chain();
    }
    close_chain();
    asm volatile("cp.async.wait_group 0;" ::: "memory");

    auto store = [&](int m, int n, float v, int z) {
        if (m >= M || n >= N) return;
        if (MODE == 2) {
            ((float*)out)[((int64_t)z * M + m) * N + n] = v;
            if (upd.w) {                                       // (one slice only) the filter is of the storage type
                T* const w = (T*)upd.w + (int64_t)m * N + n;
                *w = from_f<T>(fmaf(-upd.lr, v, to_f(*w)));
            }
        } else {
            if (bias) v += bias[n];
            if (relu) v = fmaxf(v, 0.f);
            int64_t row = m;
            if (MODE == 1 && g.stride > 1) {
                Pixel p;
                p.set(m, W, H);
                row = ((int64_t)p.n * g.h + p.h * g.stride + ph) * g.w + p.w * g.stride + pw;
            }
            ((T*)out)[row * N + n] = from_f<T>(v);
        }
    };
    // what a thread adds up of one column, or of its TN columns, meets the other threads' in shared memory, in a fixed order
    float* const red = reinterpret_cast<float*>(smem);
    auto leave_sums = [&](int row, int per_column) {          // red: [per_column][BN][sum | sum of squares]
        __syncthreads();
        if (tid < BN && n0 + tid < N) {
            float s = 0.f, q = 0.f;
            for (int r = 0; r < per_column; ++r) { s += red[(r * BN + tid) * 2]; q += red[(r * BN + tid) * 2 + 1]; }
            sums[(size_t)row * 2 * N + n0 + tid] = s;
            sums[((size_t)row * 2 + 1) * N + n0 + tid] = q;
        }
    };
    auto add = [&](float v, float& s, float& q) { const float r = to_f(from_f<T>(v)); s += r; q = fmaf(r, r, q); };
    if (cluster == 1) {
#pragma unroll
        for (int i = 0; i < TM; ++i)
#pragma unroll
            for (int j = 0; j < TN; ++j) store(m0 + m_of(i), n0 + n_of(j), sum_of(i, j), blockIdx.z);
        if (MODE == 0 && sums) {
            __syncthreads();                                  // every stage has been read
#pragma unroll
            for (int j = 0; j < TN; ++j) {
                float s = 0.f, q = 0.f;
#pragma unroll
                for (int i = 0; i < TM; ++i)
                    if (m0 + m_of(i) < M) add(sum_of(i, j), s, q);
                red[(ty * BN + n_of(j)) * 2] = s;
                red[(ty * BN + n_of(j)) * 2 + 1] = q;
            }
            leave_sums(blockIdx.x, TY);
        }
        return;
    }
    // ---- partial tiles of the cluster, added in rank order by the CTA that stores that share of the tile
    namespace cg = cooperative_groups;
    cg::cluster_group cl = cg::this_cluster();
    float* const tile = reinterpret_cast<float*>(smem);
    __syncthreads();                                          // every stage has been read
#pragma unroll
    for (int i = 0; i < TM; ++i)
#pragma unroll
        for (int j = 0; j < TN; ++j) tile[m_of(i) * BN + n_of(j)] = sum_of(i, j);
    cl.sync();
    const int rank = (int)cl.block_rank(), share = BM * BN / cluster;
    static_assert(NT % BN == 0, "a thread keeps its column of the tile");
    float sum = 0.f, sumsq = 0.f;
    for (int e = rank * share + tid; e < (rank + 1) * share; e += NT) {
        float v = 0.f;
        for (int s = 0; s < cluster; ++s) v += cl.map_shared_rank(tile, s)[e];
        store(m0 + e / BN, n0 + e % BN, v, blockIdx.z / cluster);
        if (MODE == 0 && sums && m0 + e / BN < M) add(v, sum, sumsq);
    }
    cl.sync();                                                // no CTA may leave, or use its tile's room, while it is being read
    if (MODE == 0 && sums) {
        red[tid * 2] = sum;                                   // thread tid: part tid / BN of column tid % BN
        red[tid * 2 + 1] = sumsq;
        leave_sums(blockIdx.x * cluster + rank, NT / BN);
    }
}

// ------------------------------------------------------------------------------------------------
// host side
// ------------------------------------------------------------------------------------------------
struct Plan { int tile, cluster, slices, k_per_slice; bool wide = false; };

// Tile shapes, largest first.  Modes 0 and 1 keep M (pixels) long and N (channels) as narrow as the layer; a weight
// gradient is the other way round.  (BM, BN, TM, TN)
#define CKPT_SIMT_TILES(F)                                                                                             \
    F(0, 128, 128, 8, 8) F(1, 128, 64, 8, 8) F(2, 64, 64, 8, 4) F(3, 128, 32, 8, 4) F(4, 64, 32, 4, 4) F(5, 128, 16, 4, 4) F(6, 64, 16, 4, 2)
#define CKPT_SIMT_TILES_W(F)                                                                                           \
    F(0, 128, 128, 8, 8) F(1, 64, 128, 8, 8) F(2, 64, 64, 8, 4) F(3, 32, 128, 4, 8) F(4, 32, 64, 4, 4) F(5, 16, 128, 4, 4) F(6, 16, 64, 2, 4)

Plan plan(int mode, int value_bytes, int M, int N, int K, bool vectors, bool wide = false);

template <typename T>
int launch(int mode, const ConvGeom& g, const void* a, const void* b, void* out, const float* bias, int relu, int M, int N, int K,
           bool va, bool vb, const Plan& p, const SgdUpdate& upd, cudaStream_t st, float* sums = nullptr);

}  // namespace simt
}  // namespace ckpt
