// 16-byte vector access to bf16 / float32 rows, shared by the element-wise kernels.
#pragma once
#include <cuda_bf16.h>

namespace ckpt {

template <typename T> __device__ __forceinline__ float ld(const T* p);
template <> __device__ __forceinline__ float ld<float>(const float* p) { return *p; }
template <> __device__ __forceinline__ float ld<__nv_bfloat16>(const __nv_bfloat16* p) { return __bfloat162float(*p); }
template <typename T> __device__ __forceinline__ T cvt(float v);
template <> __device__ __forceinline__ float cvt<float>(float v) { return v; }
template <> __device__ __forceinline__ __nv_bfloat16 cvt<__nv_bfloat16>(float v) { return __float2bfloat16_rn(v); }

template <typename T, int VEC>
__device__ __forceinline__ void load_vec(const T* p, float (&v)[VEC]) {
    if constexpr (VEC == 1) {
        v[0] = ld(p);
    } else if constexpr (sizeof(T) == 4) {
        float4 t = *reinterpret_cast<const float4*>(p);
        v[0] = t.x; v[1] = t.y; v[2] = t.z; v[3] = t.w;
    } else {
        uint4 t = *reinterpret_cast<const uint4*>(p);
        const __nv_bfloat162* h = reinterpret_cast<const __nv_bfloat162*>(&t);
#pragma unroll
        for (int i = 0; i < 4; ++i) { float2 f = __bfloat1622float2(h[i]); v[2 * i] = f.x; v[2 * i + 1] = f.y; }
    }
}
template <typename T, int VEC>
__device__ __forceinline__ void store_vec(T* p, const float (&v)[VEC]) {
    if constexpr (VEC == 1) {
        *p = cvt<T>(v[0]);
    } else if constexpr (sizeof(T) == 4) {
        *reinterpret_cast<float4*>(p) = make_float4(v[0], v[1], v[2], v[3]);
    } else {
        uint4 t;
        __nv_bfloat162* h = reinterpret_cast<__nv_bfloat162*>(&t);
#pragma unroll
        for (int i = 0; i < 4; ++i) h[i] = __floats2bfloat162_rn(v[2 * i], v[2 * i + 1]);
        *reinterpret_cast<uint4*>(p) = t;
    }
}

// A vector as loaded: kept packed in registers until it is used, so that many loads can be in flight
// per thread without the register cost of their unpacked form.
template <typename T, int VEC> struct RawVec { T e[VEC]; };
template <> struct RawVec<__nv_bfloat16, 8> { uint4 q; };
template <> struct RawVec<float, 4> { float4 q; };
template <typename T, int VEC>
__device__ __forceinline__ RawVec<T, VEC> load_raw(const T* p) {
    RawVec<T, VEC> r;
    if constexpr (VEC == 1) r.e[0] = *p;
    else if constexpr (sizeof(T) == 4) r.q = *reinterpret_cast<const float4*>(p);
    else r.q = *reinterpret_cast<const uint4*>(p);
    return r;
}
template <typename T, int VEC>
__device__ __forceinline__ void unpack(const RawVec<T, VEC>& r, float (&v)[VEC]) {
    if constexpr (VEC == 1) {
        v[0] = (float)r.e[0];
    } else if constexpr (sizeof(T) == 4) {
        v[0] = r.q.x; v[1] = r.q.y; v[2] = r.q.z; v[3] = r.q.w;
    } else {
        const __nv_bfloat162* h = reinterpret_cast<const __nv_bfloat162*>(&r.q);
#pragma unroll
        for (int i = 0; i < 4; ++i) { float2 f = __bfloat1622float2(h[i]); v[2 * i] = f.x; v[2 * i + 1] = f.y; }
    }
}

template <typename T, int VEC>
__device__ __forceinline__ RawVec<T, VEC> pack_raw(const float (&v)[VEC]) {
    RawVec<T, VEC> r;
    store_vec<T, VEC>(reinterpret_cast<T*>(&r), v);
    return r;
}
// 16-byte vectors as plain words (to keep them in shared memory)
template <typename R> __device__ __forceinline__ uint4 as_uint4(const R& r) { return *reinterpret_cast<const uint4*>(&r); }
template <typename T, int VEC> __device__ __forceinline__ RawVec<T, VEC> from_uint4(const uint4& u) { return *reinterpret_cast<const RawVec<T, VEC>*>(&u); }
// value k of a vector (k known at compile time)
template <typename T> __device__ __forceinline__ float element(const uint4& u, int k) {
    const int w = sizeof(T) == 2 ? k / 2 : k;
    const uint32_t x = w == 0 ? u.x : w == 1 ? u.y : w == 2 ? u.z : u.w;
    return __uint_as_float(sizeof(T) == 4 ? x : k % 2 ? x & 0xffff0000u : x << 16);
}

// sum (x + y) += v without losing what the addition rounds off (Knuth's two-sum)
__device__ __forceinline__ void two_sum(float2& sum, float v) {
    const float t = sum.x + v, b = t - sum.x;
    sum.y += (sum.x - (t - b)) + (v - b);
    sum.x = t;
}
// The same with the carry taken along in the next addition (Kahan): four operations instead of seven.  What it loses is of the order of
// a last bit of v.
__device__ __forceinline__ void carry_sum(float2& sum, float v) {
    const float y = v + sum.y, t = sum.x + y;
    sum.y = y - (t - sum.x);
    sum.x = t;
}

}  // namespace ckpt
