// links.cuh - layout and loads of the FP32, FP16 and BF16 link copies.
//
// A link of E complex entries (9, or 6 for two rows) is stored in 16-byte words of
// W = 16 / sizeof(entry) entries, word-major with the site index fastest, and the
// entries left over in planes of their own:
//   [parity][mu] { [E / W words][vs][W], [E % W entries][vs] }
// (FP32, nine entries: four words and one 8-byte plane; two rows: three words;
// 16-bit, nine entries: two words and one 4-byte plane).  One load per word instead
// of one per entry: a warp reads 512 contiguous bytes where an FP16 entry plane gave it
// 128, with 3 loads and 3 addresses per link instead of 9.  At 28^3 x 96 (Naik) the
// D_oe with FP16 storage went from 102 to 93 us (632 MB: the rate of a plain copy, 0.91 to 0.93
// of the 7.3 to 7.5 TB/s that a plain read sweep reaches); the FP32 ones stayed at HBM
// speed (181 us, 156 us with two-row Naik links).  Where the links come from L2 fewer
// loads show: 24^2 x 16 x 32 FP32 28.3 -> 25.3 us, 12^3 x 16 4.4 -> 3.3 us.
// FP64 and float-float entries are 16-byte words themselves.
#pragma once

#include <cuda_bf16.h>
#include <cuda_fp16.h>
#include <cuda_runtime.h>

namespace stag {

// Offset of entry k of site i's link inside its [parity][mu] part of E * vs entries.
template <int E, class T>
__host__ __device__ __forceinline__ size_t link_offset(int k, size_t i, size_t vs) {
    constexpr int W = 16 / (int)sizeof(T), F = E / W * W;
    return k < F ? (size_t)(k / W) * W * vs + W * i + k % W : k * vs + i;
}

struct LoadCached {
    template <class T>
    static __device__ __forceinline__ T ld(const T* p) {
        return __ldg(p);
    }
};
// read once: evicted first
struct LoadStreaming {
    template <class T>
    static __device__ __forceinline__ T ld(const T* p) {
        return __ldcs(p);
    }
};

__device__ __forceinline__ float2 half2_bits(unsigned int v) {
    return __half22float2(*reinterpret_cast<const __half2*>(&v));
}
__device__ __forceinline__ float2 bf162_bits(unsigned int v) {
    return __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(&v));
}

// The E entries of site i's link; u: its [parity][mu] part.
template <int E, class Ld = LoadCached>
__device__ __forceinline__ void load_link(float2 (&U)[9], const float2* __restrict__ u, size_t vs, size_t i) {
#pragma unroll
    for (int w = 0; w < E / 2; ++w) {
        const float4 q = Ld::ld(reinterpret_cast<const float4*>(u + (size_t)2 * w * vs) + i);
        U[2 * w] = make_float2(q.x, q.y);
        U[2 * w + 1] = make_float2(q.z, q.w);
    }
    if constexpr (E % 2 != 0) U[E - 1] = Ld::ld(u + (E - 1) * vs + i);
}
template <int E, class Ld = LoadCached>
__device__ __forceinline__ void load_link(float2 (&U)[9], const __half2* __restrict__ u, size_t vs, size_t i) {
    static_assert(E == 9, "16-bit links keep all nine entries");
#pragma unroll
    for (int w = 0; w < 2; ++w) {
        const uint4 q = Ld::ld(reinterpret_cast<const uint4*>(u + (size_t)4 * w * vs) + i);
        U[4 * w] = half2_bits(q.x);
        U[4 * w + 1] = half2_bits(q.y);
        U[4 * w + 2] = half2_bits(q.z);
        U[4 * w + 3] = half2_bits(q.w);
    }
    U[8] = half2_bits(Ld::ld(reinterpret_cast<const unsigned int*>(u + 8 * vs) + i));
}
template <int E, class Ld = LoadCached>
__device__ __forceinline__ void load_link(float2 (&U)[9], const __nv_bfloat162* __restrict__ u, size_t vs, size_t i) {
    static_assert(E == 9, "16-bit links keep all nine entries");
#pragma unroll
    for (int w = 0; w < 2; ++w) {
        const uint4 q = Ld::ld(reinterpret_cast<const uint4*>(u + (size_t)4 * w * vs) + i);
        U[4 * w] = bf162_bits(q.x);
        U[4 * w + 1] = bf162_bits(q.y);
        U[4 * w + 2] = bf162_bits(q.z);
        U[4 * w + 3] = bf162_bits(q.w);
    }
    U[8] = bf162_bits(Ld::ld(reinterpret_cast<const unsigned int*>(u + 8 * vs) + i));
}
// FP64 and float-float: an entry is a word.
template <int E, class Ld = LoadCached>
__device__ __forceinline__ void load_link(double2 (&U)[9], const double2* __restrict__ u, size_t vs, size_t i) {
#pragma unroll
    for (int k = 0; k < E; ++k) U[k] = Ld::ld(u + k * vs + i);
}
template <int E, class Ld = LoadCached>
__device__ __forceinline__ void load_link(float4 (&U)[9], const float4* __restrict__ u, size_t vs, size_t i) {
#pragma unroll
    for (int k = 0; k < E; ++k) U[k] = Ld::ld(u + k * vs + i);
}

}  // namespace stag
