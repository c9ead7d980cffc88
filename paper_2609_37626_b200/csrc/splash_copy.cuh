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
    asm volatile("ld.global.v8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
                 : "=r"(x.v[0]), "=r"(x.v[1]), "=r"(x.v[2]), "=r"(x.v[3]), "=r"(x.v[4]), "=r"(x.v[5]), "=r"(x.v[6]), "=r"(x.v[7]) : "l"(ptr) : "memory");
}
__device__ __forceinline__ void store_stream(Vec32 *ptr, const Vec32 &x) {
    asm volatile("st.global.v8.b32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};"
                 ::"l"(ptr), "r"(x.v[0]), "r"(x.v[1]), "r"(x.v[2]), "r"(x.v[3]), "r"(x.v[4]), "r"(x.v[5]), "r"(x.v[6]), "r"(x.v[7]) : "memory");
}
template <typename Vec>
__device__ __forceinline__ void load_stream(Vec &x, const Vec *ptr) { x = *ptr; }
template <typename Vec>
__device__ __forceinline__ void store_stream(Vec *ptr, const Vec &x) { *ptr = x; }

// How a move of rows is dealt out to blocks.  A row of up to one round of a block goes to a group of threads, the fewest that have it in one
// round of kCopyDepth loads each as long as there are blocks for all SMs, so a block takes several short rows side by side.  A longer one goes to one block, and from
// kCopyPartBytes on, or where the rows are fewer than the SMs can use, in parts to several.  (With a block per row, whatever its
// length, rows of 1 KB came out at the rate at which blocks start, 16,384 of them in 21 us and not in 5.3, and eight rows of 1 MB from
// eight SMs, in 23 us and not in 3.8.)
constexpr int64_t kCopyPartBytes = 80 << 10;          // (the caches' own pages: one block each)
struct RowSplit {
    int64_t vecs, per;         // vectors of a row, and of a part
    int32_t group, parts;      // threads to a row (a power of two), parts of a row
    int64_t items;             // blocks
    RowSplit(int64_t rows, int64_t row_vecs, int vec_bytes, int sm_count) : vecs(row_vecs), group(kCopyThreads), parts(1) {
        constexpr int64_t kRound = kCopyDepth * kCopyThreads;
        if (vecs <= kRound) {
            while (group > 1 && vecs <= kCopyDepth * (group / 2) && rows * (group / 2) >= 4 * (int64_t)sm_count * kCopyThreads) group /= 2;
            per = vecs;
            items = (rows + kCopyThreads / group - 1) / (kCopyThreads / group);
            return;
        }
        const int64_t needed = (vecs * vec_bytes + kCopyPartBytes - 1) / kCopyPartBytes, rounds = (vecs + kRound - 1) / kRound;
        const int64_t useful = (4 * (int64_t)sm_count + rows - 1) / rows;
        int64_t p = useful < rounds ? useful : rounds;
        if (p < needed) p = needed;
        parts = (int32_t)(p < 0x7fffffff ? p : 0x7fffffff);
        per = (vecs + parts - 1) / parts;
        items = rows * parts;
    }
};

// dst[c] = src(c) for c < vecs, by a block (kBlock) or by `group` of its threads.
template <bool kBlock, typename Vec, typename Src>
__device__ __forceinline__ void copy_row(Vec *dst, int vecs, int group, Src &&src) {
    const int step = kBlock ? kCopyThreads : group, lane = kBlock ? threadIdx.x : threadIdx.x & (group - 1);
    for (int c0 = lane; c0 < vecs; c0 += kCopyDepth * step) {
        Vec x[kCopyDepth];
#pragma unroll
        for (int u = 0; u < kCopyDepth; ++u)
            if (c0 + u * step < vecs) load_stream(x[u], src(c0 + u * step));
#pragma unroll
        for (int u = 0; u < kCopyDepth; ++u)
            if (c0 + u * step < vecs) store_stream(dst + c0 + u * step, x[u]);
    }
}

// Calls move(row, first vector, vectors) for what falls to this thread's block or group.
template <bool kBlock, typename Move>
__device__ __forceinline__ void own_row(const RowSplit &w, int64_t rows, Move &&move) {
    if constexpr (kBlock) {
        if (w.parts == 1) { move((int64_t)blockIdx.x, (int64_t)0, (int)w.vecs); return; }
        const int64_t row = blockIdx.x / (unsigned)w.parts, first = (blockIdx.x - row * w.parts) * w.per;
        if (first < w.vecs) move(row, first, (int)min(w.per, w.vecs - first));
    } else {
        const int64_t row = (int64_t)blockIdx.x * (kCopyThreads / (unsigned)w.group) + threadIdx.x / (unsigned)w.group;
        if (row < rows) move(row, (int64_t)0, (int)w.vecs);
    }
}

// the widest of 32, 16 and 2 bytes that divides all of a move's addresses, pitches and lengths (as one OR of them)
inline int copy_width(uint64_t bits) { return (bits & 31) == 0 ? 32 : (bits & 15) == 0 ? 16 : 2; }
inline uint64_t address_bits(const void *p) { return (uint64_t)reinterpret_cast<uintptr_t>(p); }

}  // namespace splash
