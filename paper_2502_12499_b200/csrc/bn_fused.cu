// Batch-norm backward in one pass over its tensors: sums, coefficients and input gradient in one cooperative kernel.
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include <algorithm>
#include <cstdint>

#include "device_flags.h"
#include "internal.h"
#include "overlap.cuh"
#include "vec.cuh"

namespace ckpt {

namespace {

constexpr int kThreads = 512, kWarps = kThreads / 32;
constexpr int kMaxWidth = 128;                       // channels per group
constexpr int kMaxSplit = 16;                        // threads that share a column of the group's partial sums
constexpr long long kWaitCycles = 4000000000LL;      // ~2 s at 2 GHz
constexpr int kStatusBarrier = 801;

struct Params {
    const void *z, *mask;
    void *dy, *dz;
    const float* stats;
    float *partial, *dgamma, *dbeta;
    unsigned* counters;          // [kBnSyncGroups] arrivals, [kBnSyncGroups] departures, zero before and after the kernel
    int* status;
    int64_t rows, rows_per_part, rows_per_step;
    double inv_rows;
    int c, width, groups, parts, relu;
    SgdUpdate gamma, beta;
};

__device__ __forceinline__ unsigned load_acquire(const unsigned* p) {
    unsigned v;
    asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
    return v;
}
__device__ __forceinline__ void copy_16(uint32_t dst, const void* src) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst), "l"(src) : "memory");
}
__device__ __forceinline__ void copy_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N> __device__ __forceinline__ void copy_wait() { asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory"); }

template <bool MASK> struct Ring {
    static constexpr int tensors = MASK ? 3 : 2;                // g, z (, mask)
    static constexpr int step_bytes = tensors * kThreads * 16;
    static constexpr int slots = 200 * 1024 / step_bytes;       // steps held in shared memory
};

// A CTA owns `width` consecutive channels of one slab of rows and walks it twice, a step being one 16-byte vector of each
// tensor per thread.  First walk: per-channel sums of g and g*z; the vectors arrive in a ring in shared memory (every
// thread copies and reads its own), `slots` steps in flight, and the last ones stay there.  The CTAs of a channel group
// then meet (they are co-resident: cooperative launch), each adds up the group's partial sums for itself, and the second
// walk writes
//   dz = scale*g - A - z*B
// backwards, first what the ring still holds, then what the L2 has read last.  HBM sees g and z once for tensors up to
// 29 MB together, and one launch replaces the sums, finalize and apply kernels and the updates of scale and shift.
// Bound by HBM (first walk at 5.5 TB/s, second at 7.2 counting L2 hits, 206 MB tensors); on small tensors by the meeting
// and the sums, about 5 us.  16 warps: 20 or 24 spill registers and measured 5-20 % slower.
// MASK: dy is first masked by mask > 0, in place (the ReLU behind a residual join).
// CLUSTER: the CTAs of a group are one cluster; they meet at its barrier and read one another's sums from shared memory
// (about 2 us less than over global memory; no co-operative launch, no counters).
template <typename T, int VEC, bool MASK, bool CLUSTER>
__global__ void __launch_bounds__(kThreads, 1) bn_bwd_fused_kernel(Params p) {
    using Rg = Ring<MASK>;
    previous_grid_done();
    next_grid_may_start();
    extern __shared__ uint4 ring[];                                  // [slot][g | z | mask][thread]
    __shared__ __align__(16) float red[kWarps * 2 * kMaxWidth];      // sums per warp; then the group's sums
    __shared__ float coef[2][kMaxWidth];
    __shared__ float sums[2 * kMaxWidth];                            // CLUSTER: this CTA's, read by its peers
    __shared__ int go;
    constexpr int U = 2;
    const int tid = threadIdx.x, warp = tid / 32, lane = tid % 32;
    const int lanes = p.width / VEC, rows_per_warp = 32 / lanes;
    const int vlane = lane % lanes, wrow = lane / lanes;
    const bool active = wrow < rows_per_warp;
    const int group = CLUSTER ? blockIdx.x / p.parts : blockIdx.x % p.groups, part = CLUSTER ? blockIdx.x % p.parts : blockIdx.x / p.groups;
    const int R = rows_per_warp * kWarps;
    const int64_t row_begin = (int64_t)part * p.rows_per_part, row_end = min(p.rows, row_begin + p.rows_per_part);
    const int steps = row_end > row_begin ? (int)((row_end - row_begin + R - 1) / R) : 0;
    const int64_t c = p.c;
    const int64_t first = row_begin + warp * rows_per_warp + wrow;
    const int mine = active && first < row_end ? (int)((row_end - first + R - 1) / R) : 0;     // this thread's vectors
    const int ch = group * p.width + (active ? vlane : 0) * VEC;
    const int64_t at = first * c + ch, hop = (int64_t)R * c;
    const T* const z = (const T*)p.z + at;
    const T* const mask = (const T*)p.mask + at;
    T* const dy = (T*)p.dy + at;
    T* const dz = (T*)p.dz + at;
    const uint32_t ring_addr = (uint32_t)__cvta_generic_to_shared(ring) + tid * 16;
    auto fetch = [&](int s, bool with_mask) {
        if (s >= 0 && s < mine) {
            const uint32_t dst = ring_addr + (uint32_t)(s % Rg::slots) * Rg::step_bytes;
            copy_16(dst, dy + s * hop);
            copy_16(dst + kThreads * 16, z + s * hop);
            if (MASK && with_mask) copy_16(dst + 2 * kThreads * 16, mask + s * hop);
        }
        copy_commit();
    };
    auto slot = [&](int s) { return ring + (size_t)(s % Rg::slots) * (Rg::step_bytes / 16) + tid; };
    // the forward output, rounded to its type, is positive: for bf16 above half of the smallest subnormal
    constexpr float kPositive = sizeof(T) == 2 ? 0x1p-134f : 0.f;
    const bool all = !p.relu;
    auto passes = [&](float v, float scale, float shift) { return all || fmaf(v, scale, shift) > kPositive; };

#pragma unroll 1
    for (int s = 0; s < Rg::slots; ++s) fetch(s, true);
    float sc[VEC], sh[VEC], s0[VEC], s1[VEC];
#pragma unroll
    for (int k = 0; k < VEC; ++k) {
        sc[k] = p.stats[2 * c + ch + k];
        sh[k] = p.stats[3 * c + ch + k];
        s0[k] = 0.f; s1[k] = 0.f;
    }
    // the values of P steps are added up before they join the running sums: shorter chains of float32 additions, and the
    // ring's reads in flight together (bf16 with two steps: the training step of 32 units of 64 channels 4 % slower; float32
    // with four: the small network of eight layers 1 %)
    constexpr int P = VEC == 8 ? 4 : 2;
#pragma unroll 1
    for (int st = 0; st < steps; st += P) {
        copy_wait<Rg::slots - P>();
        uint4 gq[P], vq[P];
#pragma unroll
        for (int u = 0; u < P; ++u) {
            gq[u] = vq[u] = make_uint4(0u, 0u, 0u, 0u);
            if (st + u < mine) {
                uint4* const held = slot(st + u);
                gq[u] = held[0];
                vq[u] = held[kThreads];
                if (MASK) {
                    float g[VEC], m[VEC];
                    unpack<T, VEC>(from_uint4<T, VEC>(gq[u]), g);
                    unpack<T, VEC>(from_uint4<T, VEC>(held[2 * kThreads]), m);
#pragma unroll
                    for (int k = 0; k < VEC; ++k) g[k] = m[k] > 0.f ? g[k] : 0.f;
                    gq[u] = as_uint4(pack_raw<T, VEC>(g));
                    held[0] = gq[u];
                    *reinterpret_cast<uint4*>(dy + (st + u) * hop) = gq[u];
                }
            }
        }
#pragma unroll
        for (int k = 0; k < VEC; ++k) {
            float g[P], gz[P / 2];
#pragma unroll
            for (int u = 0; u < P; ++u) {
                // (a blocked gradient still meets its z: a NaN or an infinity there reaches the sums)
                const float v = element<T>(vq[u], k);
                g[u] = passes(v, sc[k], sh[k]) ? element<T>(gq[u], k) : 0.f;
                gz[u / 2] = u % 2 ? fmaf(g[u], v, gz[u / 2]) : g[u] * v;
            }
            if constexpr (P == 4) {
                s0[k] += (g[0] + g[1]) + (g[2] + g[3]);
                s1[k] += gz[0] + gz[1];
            } else {
                s0[k] += g[0] + g[1];
                s1[k] += gz[0];
            }
        }
#pragma unroll
        for (int u = 0; u < P; ++u) fetch(st + u + Rg::slots, true);
    }
    // rows of a warp, then the warps, in a fixed order
    if ((lanes & (lanes - 1)) == 0) {
        for (int o = 16; o >= lanes; o >>= 1) {
#pragma unroll
            for (int k = 0; k < VEC; ++k) {
                s0[k] += __shfl_xor_sync(0xffffffffu, s0[k], o);
                s1[k] += __shfl_xor_sync(0xffffffffu, s1[k], o);
            }
        }
    } else {
        float a[VEC], b[VEC];
#pragma unroll
        for (int k = 0; k < VEC; ++k) { a[k] = s0[k]; b[k] = s1[k]; }
        for (int q = 1; q < rows_per_warp; ++q) {
#pragma unroll
            for (int k = 0; k < VEC; ++k) {
                a[k] += __shfl_sync(0xffffffffu, s0[k], vlane + q * lanes);
                b[k] += __shfl_sync(0xffffffffu, s1[k], vlane + q * lanes);
            }
        }
#pragma unroll
        for (int k = 0; k < VEC; ++k) { s0[k] = a[k]; s1[k] = b[k]; }
    }
    if (wrow == 0) {
#pragma unroll
        for (int k = 0; k < VEC; ++k) {
            red[warp * 2 * p.width + vlane * VEC + k] = s0[k];
            red[warp * 2 * p.width + p.width + vlane * VEC + k] = s1[k];
        }
    }
    __syncthreads();
    const int columns = 2 * p.width;                                 // (sum g | sum g*z) x channel
    if (tid < columns) {
        // (sums of hundreds of rows: added as two floats, four chains side by side)
        float2 part4[4] = {};
#pragma unroll 1
        for (int w = 0; w < kWarps; w += 4) {
#pragma unroll
            for (int q = 0; q < 4; ++q) two_sum(part4[q], red[(w + q) * columns + tid]);
        }
#pragma unroll
        for (int q = 1; q < 4; ++q) { two_sum(part4[0], part4[q].x); part4[0].y += part4[q].y; }
        const float a = part4[0].x + part4[0].y;
        if (CLUSTER) sums[tid] = a;
        else __stcg(p.partial + ((size_t)part * 2 + tid / p.width) * c + group * p.width + tid % p.width, a);
    }
    if (!CLUSTER) __syncthreads();
    // what the coefficients need besides the sums, fetched under the wait
    double mean = 0.0, inv = 0.0, scale = 0.0;
    float old_gamma = 0.f, old_beta = 0.f;
    if (tid < p.width) {
        const int chn = group * p.width + tid;
        mean = p.stats[chn]; inv = p.stats[c + chn]; scale = p.stats[2 * c + chn];
        if (part == 0 && p.gamma.w) old_gamma = ((const float*)p.gamma.w)[chn];
        if (part == 0 && p.beta.w) old_beta = ((const float*)p.beta.w)[chn];
    }
    if (CLUSTER) {
        asm volatile("barrier.cluster.arrive.release;" ::: "memory");
        asm volatile("barrier.cluster.wait.acquire;" ::: "memory");
    } else if (tid == 0) {
        go = 1;
        if (p.parts > 1) {
            unsigned* const arrived = p.counters + group;
            asm volatile("red.release.gpu.global.add.u32 [%0], %1;" ::"l"(arrived), "r"(1u) : "memory");
            const long long t0 = clock64();
            while (load_acquire(arrived) < (unsigned)p.parts) {
                if (clock64() - t0 > kWaitCycles) { go = 0; atomicCAS(p.status, 0, kStatusBarrier); break; }
            }
        }
    }
    if (!CLUSTER) __syncthreads();
    copy_wait<0>();
    if (!CLUSTER && !go) return;
    {
        // the group's sums over its partial rows: up to kMaxSplit threads per four columns, combined in a fixed order, each
        // sum as two floats (twice float precision; conversions to double are slow)
        float2* const pair = reinterpret_cast<float2*>(red);
        if (CLUSTER && tid < columns) {
            float x[16];
#pragma unroll
            for (int r = 0; r < 16; ++r) {
                if (r >= p.parts) break;
                uint32_t at;
                asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(at) : "r"((uint32_t)__cvta_generic_to_shared(sums + tid)), "r"(r));
                asm volatile("ld.shared::cluster.f32 %0, [%1];" : "=f"(x[r]) : "r"(at) : "memory");
            }
            float2 a = {};
#pragma unroll
            for (int r = 0; r < 16; ++r)
                if (r < p.parts) two_sum(a, x[r]);
            pair[tid] = a;
        }
        const int quads = columns / 4, split = CLUSTER ? 1 : min(min(kThreads / quads, kMaxSplit), p.parts), quad = tid % quads, q = tid / quads;
        if (!CLUSTER && q < split) {
            const int col = quad * 4;
            const float* const src = p.partial + (size_t)(col / p.width) * c + group * p.width + col % p.width;
            float2 a[4] = {};
            constexpr int B = 10;                                    // loads in flight: all of them in the usual case
            for (int b0 = q; b0 < p.parts; b0 += B * split) {
                float4 x[B];
#pragma unroll
                for (int b = 0; b < B; ++b)
                    if (b0 + b * split < p.parts) x[b] = __ldcg(reinterpret_cast<const float4*>(src + (size_t)(b0 + b * split) * 2 * c));
#pragma unroll
                for (int b = 0; b < B; ++b)
                    if (b0 + b * split < p.parts) { two_sum(a[0], x[b].x); two_sum(a[1], x[b].y); two_sum(a[2], x[b].z); two_sum(a[3], x[b].w); }
            }
#pragma unroll
            for (int k = 0; k < 4; ++k) pair[q * columns + col + k] = a[k];
        }
        __syncthreads();
        if (CLUSTER) asm volatile("barrier.cluster.arrive.release;" ::: "memory");      // this CTA has read its peers' sums
        if (!CLUSTER && tid == 0 && p.parts > 1) {
            // the last one to leave puts the counters back as they were found
            if (atomicAdd(p.counters + kBnSyncGroups + group, 1u) == (unsigned)p.parts - 1u) { p.counters[group] = 0u; p.counters[kBnSyncGroups + group] = 0u; }
        }
        if (tid < p.width) {
            float2 s2 = {}, gz2 = {};
            for (int k = 0; k < split; ++k) {
                const float2 a = pair[k * columns + tid], b = pair[k * columns + p.width + tid];
                two_sum(s2, a.x); s2.y += a.y;
                two_sum(gz2, b.x); gz2.y += b.y;
            }
            const double s = (double)s2.x + s2.y, gz = (double)gz2.x + gz2.y;
            const int chn = group * p.width + tid;
            const double gx = inv * (gz - mean * s);                 // sum g*xhat
            // dz = scale*g - k1 - xhat*k2 with k1 = scale*dbeta/rows, k2 = scale*dgamma/rows, regrouped
            const double k1 = scale * s * p.inv_rows, k2 = scale * gx * p.inv_rows;
            coef[0][tid] = (float)(k1 - mean * inv * k2);
            coef[1][tid] = (float)(inv * k2);
            if (part == 0) {
                p.dbeta[chn] = (float)s;
                p.dgamma[chn] = (float)gx;
                if (p.gamma.w) ((float*)p.gamma.w)[chn] = fmaf(-p.gamma.lr, (float)gx, old_gamma);
                if (p.beta.w) ((float*)p.beta.w)[chn] = fmaf(-p.beta.lr, (float)s, old_beta);
            }
        }
        __syncthreads();
    }
    if (!CLUSTER && !active) return;
    float ca[VEC], cb[VEC];
#pragma unroll
    for (int k = 0; k < VEC; ++k) { ca[k] = coef[0][vlane * VEC + k]; cb[k] = coef[1][vlane * VEC + k]; }
    // the walk backwards starts at step `steps - 1` for every thread, so that a step keeps its slot
#pragma unroll 1
    for (int st = steps - 1; st >= 0; st -= U) {
        copy_wait<Rg::slots - U>();
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const int s = st - u;
            if (s >= 0 && s < mine) {
                const uint4* const held = slot(s);
                float v[VEC], g[VEC], o[VEC];
                unpack<T, VEC>(from_uint4<T, VEC>(held[0]), g);
                unpack<T, VEC>(from_uint4<T, VEC>(held[kThreads]), v);
#pragma unroll
                for (int k = 0; k < VEC; ++k) {
                    const float gi = passes(v[k], sc[k], sh[k]) ? g[k] : 0.f;
                    o[k] = fmaf(-v[k], cb[k], fmaf(sc[k], gi, -ca[k]));
                }
                store_vec<T, VEC>(dz + s * hop, o);
            }
        }
#pragma unroll
        for (int u = 0; u < U; ++u) fetch(st - u - Rg::slots, false);
    }
    if (CLUSTER) asm volatile("barrier.cluster.wait.acquire;" ::: "memory");           // no CTA leaves while a peer reads its sums
}

// What the device holds at once, every CTA with its whole ring: clusters of 16, 8 and 4 CTAs, and CTAs.  Asked once per device
// and instantiation (a cluster lies within a GPC; B200: 7, 15, 33 and 148).
struct Resident { int clusters[3], ctas; };
constexpr int kClusterSizes[3] = {16, 8, 4};
template <typename T, int VEC, bool MASK>
int ask(Resident* r) {
    static Resident known[kMaxDevices];
    static DeviceFlags asked;
    int dev = 0, sms = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return cuda_fail(e, "asking for the device");
    return asked.once(dev, known, r, [&](Resident* out) {
        constexpr int smem = Ring<MASK>::slots * Ring<MASK>::step_bytes;
        const auto in_clusters = bn_bwd_fused_kernel<T, VEC, MASK, true>;
        const auto cooperative = bn_bwd_fused_kernel<T, VEC, MASK, false>;
        e = cudaFuncSetAttribute(in_clusters, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
        if (e == cudaSuccess) e = cudaFuncSetAttribute(cooperative, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
        if (e == cudaSuccess) e = cudaFuncSetAttribute(in_clusters, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
        for (int i = 0; i < 3 && e == cudaSuccess; ++i) {
            cudaLaunchConfig_t cfg = {};
            cfg.gridDim = dim3((unsigned)kClusterSizes[i]); cfg.blockDim = dim3(kThreads); cfg.dynamicSmemBytes = smem;
            cudaLaunchAttribute attr;
            attr.id = cudaLaunchAttributeClusterDimension;
            attr.val.clusterDim.x = (unsigned)kClusterSizes[i]; attr.val.clusterDim.y = 1; attr.val.clusterDim.z = 1;
            cfg.attrs = &attr; cfg.numAttrs = 1;
            // (a size that the device does not have is no error: none of it is held)
            if (cudaOccupancyMaxActiveClusters(&out->clusters[i], in_clusters, &cfg) != cudaSuccess) { out->clusters[i] = 0; cudaGetLastError(); }
        }
        if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
        if (e == cudaSuccess) e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&out->ctas, cooperative, kThreads, smem);
        out->ctas *= sms;
        return e == cudaSuccess ? CKPT_OK : cuda_fail(e, "preparing the fused batch-norm backward");
    });
}
int resident(int dtype, bool mask, Resident* r) {
    if (dtype == CKPT_DTYPE_BF16) return mask ? ask<__nv_bfloat16, 8, true>(r) : ask<__nv_bfloat16, 8, false>(r);
    return mask ? ask<float, 4, true>(r) : ask<float, 4, false>(r);
}

template <typename T, int VEC>
int launch(Params& p, bool cluster, cudaStream_t st) {
    const int64_t steps = (p.rows_per_part + p.rows_per_step - 1) / p.rows_per_step;
    const size_t smem = p.mask ? (size_t)std::min<int64_t>(steps, Ring<true>::slots) * Ring<true>::step_bytes
                               : (size_t)std::min<int64_t>(steps, Ring<false>::slots) * Ring<false>::step_bytes;
    cudaError_t e;
    if (cluster) {
        cudaLaunchConfig_t cfg = {};
        cfg.gridDim = dim3((unsigned)(p.groups * p.parts)); cfg.blockDim = dim3(kThreads); cfg.dynamicSmemBytes = smem; cfg.stream = st;
        cudaLaunchAttribute attr[2];
        attr[0].id = cudaLaunchAttributeClusterDimension;
        attr[0].val.clusterDim.x = (unsigned)p.parts; attr[0].val.clusterDim.y = 1; attr[0].val.clusterDim.z = 1;
        cfg.attrs = attr; cfg.numAttrs = 1;
        start_early(&cfg, attr, Start::ON_STREAMS);
        e = p.mask ? cudaLaunchKernelEx(&cfg, bn_bwd_fused_kernel<T, VEC, true, true>, p) : cudaLaunchKernelEx(&cfg, bn_bwd_fused_kernel<T, VEC, false, true>, p);
    } else {
        void* args[] = {&p};
        const void* kernel = p.mask ? (const void*)bn_bwd_fused_kernel<T, VEC, true, false> : (const void*)bn_bwd_fused_kernel<T, VEC, false, false>;
        e = cudaLaunchCooperativeKernel(kernel, dim3((unsigned)(p.groups * p.parts)), dim3(kThreads), args, smem, st);
    }
    if (e != cudaSuccess) return cuda_fail(e, "launching the fused batch-norm backward");
    CKPT_LAUNCH_CHECK_NAMED("bn_bwd_fused_kernel", "batch-norm backward (fused)");
    return CKPT_OK;
}

// Channels per group: whole 128-byte lines where the channel count has such a divisor, twice that for very wide rows
// (fewer groups leave more CTAs to each).  0 = no usable split.
int pick_width(int c, int vec) {
    const int most = std::min(c >= 2048 ? 128 : 64, 32 * vec);
    for (int w = std::min(c, most); w >= vec; --w)
        if (c % w == 0 && w % vec == 0 && (w >= 32 || w == c)) return w;
    for (int w = most + 1; w <= std::min(kMaxWidth, 32 * vec); ++w)
        if (c % w == 0 && w % vec == 0) return w;
    return 0;
}

// How the rows of a tensor are divided.
struct Split { BnForm form; int width, groups, parts; int64_t rows_per_part, rows_per_step; };
Split divide(int dtype, int64_t rows, int c, bool mask, const Resident& r) {
    Split s = {};
    const int vec = dtype == CKPT_DTYPE_BF16 ? 8 : 4;
    s.width = c % vec ? 0 : pick_width(c, vec);
    if (s.width == 0 || c / s.width > kBnSyncGroups) return s;
    s.groups = c / s.width;
    const int64_t R = (32 / (s.width / vec)) * kWarps;               // rows per step of a CTA
    s.rows_per_step = R;
    // One cluster per group where its CTAs get no more than 0.6 of their rings and all clusters find their SMs at once.
    // Fewer CTAs then cost less than the meeting over global memory (with a 2 us memset: 3003 x 256 12.4 -> 10.4 us,
    // 882 x 2048 14.4 -> 12.4, 6272 x 256 14.3 -> 12.5; above the line 8192 x 256 14.3 either way, 11025 x 128 14.4 -> 16.0).
    for (int i = 0; i < 3; ++i) {
        if (r.clusters[i] < s.groups) continue;
        if (rows * 10 > (mask ? Ring<true>::slots : Ring<false>::slots) * R * kClusterSizes[i] * 6) break;
        s.form = BnForm::clusters;
        // no more CTAs than have a step each
        for (s.parts = kClusterSizes[i]; s.parts > 1 && (int64_t)(s.parts / 2) * R >= rows; s.parts /= 2) {}
        s.rows_per_part = (rows + s.parts - 1) / s.parts;
        return s;
    }
    if (r.ctas < s.groups) return s;                                 // the CTAs of the grid wait for one another
    s.form = BnForm::cooperative;
    s.parts = (int)std::max<int64_t>(1, std::min<int64_t>(r.ctas / s.groups, (2 * rows + R - 1) / R));
    s.rows_per_part = (rows + s.parts - 1) / s.parts;
    s.parts = (int)((rows + s.rows_per_part - 1) / s.rows_per_part);
    return s;
}

}  // namespace

// On larger tensors the separate passes stream as fast and their blocks are balanced by the hardware (bf16 with its own
// launches, us, three kernels -> one: 25088 x 256 23.1 -> 20.5, 6272 x 2048 62.4 -> 26.7, 100352 x 512 (103 MB) 99 -> 94,
// 401408 x 256 (206 MB) 178 -> 181, 3211264 x 64 (411 MB) 317 -> 354).  With a mask the pass it saves decides.
constexpr int64_t kLargest = 128 << 20;

BnForm bn_backward_form(int dtype, int64_t rows, int c, const void* dy, const void* z, const void* mask, const void* dz) {
    if (((uintptr_t)dy | (uintptr_t)z | (uintptr_t)mask | (uintptr_t)dz) & 15u) return BnForm::separate;
    if (!mask && rows * c * dtype_size(dtype) > kLargest) return BnForm::separate;
    Resident r;
    return resident(dtype, mask != nullptr, &r) == CKPT_OK ? divide(dtype, rows, c, mask != nullptr, r).form : BnForm::separate;
}

void bn_selftest_split(int dtype, int64_t rows, int c, bool mask, const int* held, int* split) {
    const Split s = divide(dtype, rows, c, mask, Resident{{held[0], held[1], held[2]}, held[3]});
    split[0] = (int)s.form; split[1] = s.groups; split[2] = s.parts;
}

int bn_backward_fused(int dtype, int64_t rows, int c, void* dy, const void* z, const float* stats, int relu, void* dz, float* dgamma,
                      float* dbeta, float* partial, const BnBackwardExtra& ex, void* stream) {
    Resident r;
    int rc = resident(dtype, ex.mask != nullptr, &r);
    if (rc) return rc;
    const Split s = divide(dtype, rows, c, ex.mask != nullptr, r);
    if (s.form == BnForm::separate) { set_error("the fused batch-norm backward does not take this tensor"); return CKPT_E_UNSUPPORTED; }
    Params p;
    p.z = z; p.mask = ex.mask; p.dy = dy; p.dz = dz; p.stats = stats; p.partial = partial; p.dgamma = dgamma; p.dbeta = dbeta;
    p.counters = ex.counters; p.status = ex.status; p.rows = rows; p.inv_rows = 1.0 / (double)rows; p.c = c; p.relu = relu;
    p.gamma = ex.gamma; p.beta = ex.beta;
    p.width = s.width; p.groups = s.groups; p.parts = s.parts; p.rows_per_part = s.rows_per_part; p.rows_per_step = s.rows_per_step;
    const bool cluster = s.form == BnForm::clusters;
    return dtype == CKPT_DTYPE_BF16 ? launch<__nv_bfloat16, 8>(p, cluster, (cudaStream_t)stream) : launch<float, 4>(p, cluster, (cudaStream_t)stream);
}

}  // namespace ckpt
