// Copies of long rows of bytes by a block, for the kernels that only move data (page migration, DOP layout changes).
//
// Bound by HBM, half reads and half writes.  What counts is bytes in flight: a block of 256 threads takes a row in rounds
// of kCopyDepth 32-byte loads per thread, all issued before the first store, four blocks to an SM (160 KB in flight); one
// 16-byte load and its store at a time, eight blocks to an SM, moved 5.4 to 5.9 TB/s.
#pragma once

#include "splash_common.cuh"

namespace splash {

constexpr int kCopyThreads = 256;
constexpr int kCopyDepth = 5;               // loads in flight per thread

struct alignas(32) Vec32 { uint32_t v[8]; };

__device__ __forceinline__ void load_stream(Vec32 &x, const Vec32 *ptr) {
    asm volatile("ld.global.nc.v8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
                 : "=r"(x.v[0]), "=r"(x.v[1]), "=r"(x.v[2]), "=r"(x.v[3]), "=r"(x.v[4]), "=r"(x.v[5]), "=r"(x.v[6]), "=r"(x.v[7]) : "l"(ptr));
}
__device__ __forceinline__ void store_stream(Vec32 *ptr, const Vec32 &x) {
    asm volatile("st.global.v8.b32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};"
                 ::"l"(ptr), "r"(x.v[0]), "r"(x.v[1]), "r"(x.v[2]), "r"(x.v[3]), "r"(x.v[4]), "r"(x.v[5]), "r"(x.v[6]), "r"(x.v[7]) : "memory");
}
template <typename Vec>
__device__ __forceinline__ void load_stream(Vec &x, const Vec *ptr) { x = __ldg(ptr); }
template <typename Vec>
__device__ __forceinline__ void store_stream(Vec *ptr, const Vec &x) { *ptr = x; }

// dst[c] = src(c) for c < vecs, by the kCopyThreads threads of a block; src gives the address of vector c.
template <typename Vec, typename Src>
__device__ __forceinline__ void copy_row(Vec *dst, int vecs, Src &&src) {
    for (int c0 = threadIdx.x; c0 < vecs; c0 += kCopyDepth * kCopyThreads) {
        Vec x[kCopyDepth];
#pragma unroll
        for (int u = 0; u < kCopyDepth; ++u)
            if (c0 + u * kCopyThreads < vecs) load_stream(x[u], src(c0 + u * kCopyThreads));
#pragma unroll
        for (int u = 0; u < kCopyDepth; ++u)
            if (c0 + u * kCopyThreads < vecs) store_stream(dst + c0 + u * kCopyThreads, x[u]);
    }
}

// the widest of 32, 16 and 2 bytes that divides all of a move's addresses, pitches and lengths (as one OR of them)
inline int copy_width(uint64_t bits) { return (bits & 31) == 0 ? 32 : (bits & 15) == 0 ? 16 : 2; }
inline uint64_t address_bits(const void *p) { return (uint64_t)reinterpret_cast<uintptr_t>(p); }

}  // namespace splash
