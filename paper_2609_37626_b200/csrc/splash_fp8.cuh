// Building blocks shared by the e4m3 decode kernels: 8-bit MMA issue, conversions, swizzle.
#pragma once

#include <cuda_fp16.h>

#include "splash_umma.cuh"

namespace splash {
namespace umma {

__host__ __device__ constexpr uint32_t make_idesc_e4m3(int M, int N, int a_mn_major, int b_e5m2 = 0, int b_mn_major = 0,
                                                        int a_e5m2 = 0) {
    // fp32 accumulate (bit 4); A / B formats E4M3 (= 0) or E5M2 (= 1) in bits 7..9 / 10..12
    return (1u << 4) | ((uint32_t)a_e5m2 << 7) | ((uint32_t)b_e5m2 << 10) | ((uint32_t)a_mn_major << 15) |
           ((uint32_t)b_mn_major << 16) | ((uint32_t)(N >> 3) << 17) | ((uint32_t)(M >> 4) << 24);
}

// Issued by the lane with `elected` != 0 (elect_one of a converged warp whose operands are uniform; 1 in a branch of one lane).
__device__ __forceinline__ void umma_e4m3(uint32_t elected, uint32_t d_tmem, uint64_t a_desc, uint64_t b_desc, uint32_t idesc, uint32_t accumulate) {
    asm volatile(
        "{\n\t.reg .pred p, q;\n\t"
        "setp.ne.b32 p, %4, 0;\n\t"
        "setp.ne.b32 q, %5, 0;\n\t"
        "@q tcgen05.mma.cta_group::1.kind::f8f6f4 [%0], %1, %2, %3, p;\n\t}"
        ::"r"(d_tmem), "l"(a_desc), "l"(b_desc), "r"(idesc), "r"(accumulate), "r"(elected) : "memory");
}

__device__ __forceinline__ void bulk_load(uint32_t dst, const void *src, uint32_t bytes, uint32_t bar) {
    asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];"
                 ::"r"(dst), "l"(src), "r"(bytes), "r"(bar) : "memory");
}

// two floats -> two e4m3 bytes (first argument in the low byte), round to nearest, saturating
__device__ __forceinline__ uint16_t to_e4m3x2(float lo, float hi) {
    uint16_t r;
    asm("cvt.rn.satfinite.e4m3x2.f32 %0, %1, %2;" : "=h"(r) : "f"(hi), "f"(lo));
    return r;
}
__device__ __forceinline__ uint16_t to_e5m2x2(float lo, float hi) {
    uint16_t r;
    asm("cvt.rn.satfinite.e5m2x2.f32 %0, %1, %2;" : "=h"(r) : "f"(hi), "f"(lo));
    return r;
}
__device__ __forceinline__ float2 from_e4m3x2(uint16_t v) {
    uint32_t h2;
    asm("cvt.rn.f16x2.e4m3x2 %0, %1;" : "=r"(h2) : "h"(v));
    __half2 h = *reinterpret_cast<__half2 *>(&h2);
    return __half22float2(h);
}
// The same split in packed f16 arithmetic: two floats -> (e4m3 pair, e5m2 pair of the residuals), five instructions.
// The detour through f16 (11 significant bits, values below 65,504) costs nothing that the 2-bit mantissa of the
// residual does not already cost; the residual itself is exact in f16.
__device__ __forceinline__ void split_e4m3_e5m2_x2(float lo, float hi, uint16_t &main, uint16_t &rest) {
    uint32_t h2, back, res;
    asm("cvt.rn.f16x2.f32 %0, %1, %2;" : "=r"(h2) : "f"(hi), "f"(lo));
    asm("cvt.rn.satfinite.e4m3x2.f16x2 %0, %1;" : "=h"(main) : "r"(h2));
    asm("cvt.rn.f16x2.e4m3x2 %0, %1;" : "=r"(back) : "h"(main));
    asm("sub.rn.f16x2 %0, %1, %2;" : "=r"(res) : "r"(h2), "r"(back));
    asm("cvt.rn.satfinite.e5m2x2.f16x2 %0, %1;" : "=h"(rest) : "r"(res));
}
// Two floats -> (e4m3 pair, e4m3 pair of the residuals) in packed f16 arithmetic, for the query operands: the value
// passes through f16 (11 significant bits against the 8 of the bf16 query it comes from), the residual is exact in f16.
__device__ __forceinline__ void split_e4m3_e4m3_x2(float lo, float hi, uint16_t &main, uint16_t &rest) {
    uint32_t h2, back, res;
    asm("cvt.rn.f16x2.f32 %0, %1, %2;" : "=r"(h2) : "f"(hi), "f"(lo));
    asm("cvt.rn.satfinite.e4m3x2.f16x2 %0, %1;" : "=h"(main) : "r"(h2));
    asm("cvt.rn.f16x2.e4m3x2 %0, %1;" : "=r"(back) : "h"(main));
    asm("sub.rn.f16x2 %0, %1, %2;" : "=r"(res) : "r"(h2), "r"(back));
    asm("cvt.rn.satfinite.e4m3x2.f16x2 %0, %1;" : "=h"(rest) : "r"(res));
}
// Two floats -> (e4m3 pair, e4m3 pair of 16 x the residuals): the residual of an e4m3 rounding is at most 2^-4 of
// the value, so 16 x residual fits the format whenever the value does, and keeps three significant bits.  For kernels
// that accumulate the two terms separately and add them as hi + lo / 16.
__device__ __forceinline__ void split_e4m3_e4m3x16_x2(float lo, float hi, uint16_t &main, uint16_t &rest) {
    uint32_t h2, back, res;
    asm("cvt.rn.f16x2.f32 %0, %1, %2;" : "=r"(h2) : "f"(hi), "f"(lo));
    asm("cvt.rn.satfinite.e4m3x2.f16x2 %0, %1;" : "=h"(main) : "r"(h2));
    asm("cvt.rn.f16x2.e4m3x2 %0, %1;" : "=r"(back) : "h"(main));
    asm("sub.rn.f16x2 %0, %1, %2;" : "=r"(res) : "r"(h2), "r"(back));
    asm("mul.rn.f16x2 %0, %1, %2;" : "=r"(res) : "r"(res), "r"(0x4C004C00u));     // x 16
    asm("cvt.rn.satfinite.e4m3x2.f16x2 %0, %1;" : "=h"(rest) : "r"(res));
}
__device__ __forceinline__ float fast_log2(float x) {
    float y;
    asm("lg2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}
__device__ __forceinline__ float fast_rcp(float x) {
    float y;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}

// ---- query operands ---------------------------------------------------------------
// The rows of kHeads heads arrive by one TMA load as bf16, [9 chunks][kHeads rows][128 B] in the 128-byte swizzle, and become the two
// 8-bit terms in place: the 1,024 bytes of eight rows of a chunk are then eight rows of 64 hi bytes and eight of 64 lo bytes in
// the 64-byte swizzle.  A converter warp has kHeads / kWarps rows, whole groups of eight, so that what it overwrites is its own; a lane has a
// row and every kParts-th chunk, eight neighbouring lanes eight neighbouring rows (no bank conflicts).
// (The rows were loaded from global memory into registers, twice over, for the maximum and for the conversion, in seven round trips where the
// registers of 128 threads hold a quarter of them: 6.4 us from the plan to the operands of a call's first request on 128 heads, now 4.2.  For 16 or 32
// heads, whose rows fit those registers at once, that is the faster way: eight layers of 8 requests 123 us, 127 this way.)
template <int kHeads, int kWarps>
struct QueryRows {
    static constexpr int kRows = kHeads / kWarps, kParts = 32 / kRows;
    static constexpr uint32_t kBytes = kHeads * kDQK * 2;
    static_assert(kRows % 8 == 0 && 32 % kRows == 0, "whole groups of eight rows");
    uint8_t *const operand;
    const uint8_t *src;          // the row as it came
    uint8_t *dst;                // its hi bytes
    int row, part;
    __device__ __forceinline__ QueryRows(uint8_t *operand_, int warp, int lane) : operand(operand_) {
        row = warp * kRows + lane % kRows; part = lane / kRows;
        src = operand + row * 128;
        dst = operand + (row >> 3) * 1024 + (row & 7) * 64;
    }
    // What the TMA load delivers, this warp's rows of it, without a tensor map: row r of the slice's `live` rows at q + r * stride (elements),
    // zeros behind them.  All of a lane's copies are in flight at once.  (Read into registers where they are used, for the maximum and
    // again for the terms, the rows were ten round trips: 512 requests of 200 to 1,500 tokens with one query for all, 128 heads, 166 us, now 138.)
    // Out of line, or the kernel's other roles pay for its registers: 8 requests on 128 heads 26.2 us instead of 25.8, whatever their rows come by.
    __device__ __noinline__ void copy_by_hand(const uint16_t *q, int64_t stride, int live, int lane) const {
        const int first = row - lane % kRows;
#pragma unroll 4
        for (int i = lane; i < kRows * 72; i += 32) {
            const int r = first + i / 72, v = i % 72;
            uint8_t *const to = operand + (v >> 3) * (kHeads * 128) + r * 128 + (((v ^ r) & 7) << 4);
            if (r < live) asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(smem_u32(to)), "l"(q + (int64_t)r * stride + v * 8) : "memory");
            else *reinterpret_cast<uint4 *>(to) = make_uint4(0u, 0u, 0u, 0u);
        }
        asm volatile("cp.async.wait_all;" ::: "memory");
        __syncwarp();
    }
    __device__ __forceinline__ void load(uint4 (&x)[8], int c) const {
#pragma unroll
        for (int j = 0; j < 8; ++j) x[j] = *reinterpret_cast<const uint4 *>(src + c * (kHeads * 128) + (((j ^ row) & 7) << 4));
    }
    // largest magnitude of the row (a NaN is passed over), the same in the lanes that share it.
    __device__ __forceinline__ float largest() const {
        uint32_t m = 0;
#pragma unroll 1
        for (int c = part; c < 9; c += kParts) {
            uint4 x[8];
            load(x, c);
#pragma unroll
            for (int j = 0; j < 8; ++j) {
                const uint32_t w[4] = {x[j].x, x[j].y, x[j].z, x[j].w};
#pragma unroll
                for (int k = 0; k < 4; ++k) asm("max.bf16x2 %0, %0, %1;" : "+r"(m) : "r"(w[k] & 0x7fff7fffu));
            }
        }
        float v = fmaxf(__uint_as_float(m << 16), __uint_as_float(m & 0xffff0000u));
#pragma unroll
        for (int o = kRows; o < 32; o <<= 1) v = fmaxf(v, __shfl_xor_sync(0xffffffffu, v, o));
        return v;
    }
    __device__ __forceinline__ void split(float inv) const {
#pragma unroll 1
        for (int i = 0; i < (9 + kParts - 1) / kParts; ++i) {
            const int c = part + i * kParts;
            uint4 x[8];
            if (c < 9) load(x, c);
            __syncwarp();                 // the eight rows have been read
            if (c < 9) {
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    uint32_t hi[4], lo[4];
#pragma unroll
                    for (int e = 0; e < 2; ++e) {
                        const uint4 v = x[2 * j + e];
                        const uint32_t w[4] = {v.x, v.y, v.z, v.w};
                        uint16_t h[4], l[4];
#pragma unroll
                        for (int k = 0; k < 4; ++k)
                            split_e4m3_e4m3_x2(__uint_as_float(w[k] << 16) * inv, __uint_as_float(w[k] & 0xffff0000u) * inv, h[k], l[k]);
                        hi[2 * e] = (uint32_t)h[0] | ((uint32_t)h[1] << 16); hi[2 * e + 1] = (uint32_t)h[2] | ((uint32_t)h[3] << 16);
                        lo[2 * e] = (uint32_t)l[0] | ((uint32_t)l[1] << 16); lo[2 * e + 1] = (uint32_t)l[2] | ((uint32_t)l[3] << 16);
                    }
                    uint8_t *const at = dst + c * (kHeads * 128) + (((j ^ (row >> 1)) & 3) << 4);
                    *reinterpret_cast<uint4 *>(at) = make_uint4(hi[0], hi[1], hi[2], hi[3]);
                    *reinterpret_cast<uint4 *>(at + 512) = make_uint4(lo[0], lo[1], lo[2], lo[3]);
                }
            }
        }
    }
};

// The map of those loads, over the heads below head_end (a box reads zeros past them).  False where the strides are none that a map can
// state: the kernel then loads the rows by hand, and the call has not failed.
inline bool make_query_map(CUtensorMap *map, const DecodeParams &p, uint32_t heads) {
    const int64_t limit = (int64_t)1 << 39;          // in elements of two bytes
    if (p.q_stride_head >= limit || (p.B > 1 && (p.q_stride_request <= 0 || p.q_stride_request >= limit))) return false;
    // (one request: any stride that a map takes)
    return encode_map_4d(map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, CU_TENSOR_MAP_SWIZZLE_128B, p.q, (uint64_t)p.head_end, (uint64_t)p.B,
                         (uint64_t)p.q_stride_head * 2, 128, (uint64_t)(p.B > 1 ? p.q_stride_request : p.q_stride_head) * 2, heads, 9) == CUDA_SUCCESS;
}

}  // namespace umma
}  // namespace splash
