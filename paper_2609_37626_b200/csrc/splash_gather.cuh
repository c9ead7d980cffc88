// Sparse decode: the rows an indexer selected for each request -- 656 bytes: 512 e4m3 latent codes, four float scales,
// one per 128 latent dims, 64 bf16 rope values (Sec. 5 setup, App. B payload) -- fetched, dequantised (code x block scale,
// rounded to bf16) and written into a decode CTA's shared-memory stages in the layout that the TMA unit gives dense pages.
//
// Eight warps of every decode CTA do it, so a listed row crosses HBM once and its 1,152 dequantised bytes never leave the SM.
// 64 requests x 2,048 tokens on 128 heads: 82 us a call.  (A kernel in front of the decode that wrote them to a dense cache took
// 46 us of 107.  The same warps writing to a ring of pages in L2 for TMA loads: 143 us, the fences between a warp's
// global stores and the copy engine's reads cost 3,000 cycles a tile.)  What bounds it
// is the gathering warps' own way round their loop: of 3,650 cycles a tile (CTA 0 of that call, traced) 1,840 go with the own rows, 735 with the
// other CTA's columns and 1,080 with the loads and addresses of the next, and none with waiting, for a stage has been free for 2,700 cycles when they
// come to it and QK^T has long retired.  No one part of the work is all of it: 74 us without the conversions, 82 without the row loads.
// (One tile of lag more or less: 5 and 13 us slower.)  A register is loaded
// again for the next tile as soon as it has been converted, and the addresses of a warp's next 32 rows -- list entry, page id, row -- are resolved one
// link of that chain per step.  The loop has one body, not unrolled over tiles: the CTA's warps are in loops of five kinds,
// and with 45 KB of code in this one they waited for instructions.
#pragma once

#include <cuda_bf16.h>

#include "splash_fp8.cuh"

namespace splash {

constexpr int kSparseRowBytes = 656;
constexpr int kGatherWarps = 8;                // of a decode CTA

namespace gather {

// What a lane knows about a row: its address, or one of these
constexpr unsigned long long kSkip = 0, kPoison = 1;           // no such row (zeros); a bad list entry, page id or count (NaN)

// 16 bytes at a global address (a plain load of an address made from an integer would be a generic one)
__device__ __forceinline__ uint4 load_global16(unsigned long long at) {
    uint4 v;
    asm volatile("ld.global.v4.b32 {%0, %1, %2, %3}, [%4];" : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "l"(at) : "memory");
    return v;
}

// 16 codes of a row or 16 bytes of its rope part
__device__ __forceinline__ uint4 load16(unsigned long long row, uint32_t offset, uint32_t poison) {
    if (row > kPoison) return load_global16(row + offset);
    const uint32_t fill = row == kPoison ? poison : 0u;
    return make_uint4(fill, fill, fill, fill);
}
constexpr uint32_t kPoisonCodes = 0x7f7f7f7fu, kPoisonRope = 0x7fc07fc0u;      // e4m3 and bf16 NaN

// 4 codes (one 32-bit word) times a scale -> 4 bf16 (two words)
__device__ __forceinline__ uint2 dequant4(uint32_t w, float s) {
    uint32_t r[2];
#pragma unroll
    for (int i = 0; i < 2; ++i) {
        const float2 a = umma::from_e4m3x2((uint16_t)(w >> (16 * i)));
        unsigned long long x, y;
        asm("mov.b64 %0, {%1, %2};" : "=l"(x) : "f"(a.x), "f"(a.y));
        asm("mov.b64 %0, {%1, %1};" : "=l"(y) : "f"(s));
        asm("mul.rn.f32x2 %0, %0, %1;" : "+l"(x) : "l"(y));
        float lo, hi;
        asm("mov.b64 {%0, %1}, %2;" : "=f"(lo), "=f"(hi) : "l"(x));
        r[i] = umma::pack_bf16x2(lo, hi);
    }
    return make_uint2(r[0], r[1]);
}

// 16 codes x scale -> 32 bytes of a 128-byte-swizzled slab row: 16-byte units `unit` and `unit + 1` (unit even)
__device__ __forceinline__ void dequant16(uint4 codes, float s, uint8_t *slab_row, int r, int unit) {
    const uint2 a = dequant4(codes.x, s), b = dequant4(codes.y, s), c = dequant4(codes.z, s), d = dequant4(codes.w, s);
    *reinterpret_cast<uint4 *>(slab_row + ((unit ^ (r & 7)) << 4)) = make_uint4(a.x, a.y, b.x, b.y);
    *reinterpret_cast<uint4 *>(slab_row + (((unit + 1) ^ (r & 7)) << 4)) = make_uint4(c.x, c.y, d.x, d.y);
}

// Resolves the rows that a warp will need next: lane l those of tile l / kShare of the group, row first + l % kShare of its
// kPage rows, and (kPeer) the row 32 further or nearer, which the other CTA of a pair multiplies.
template <int kShare, bool kPeer, typename Iter>
struct Resolver {
    static constexpr int kTiles = 32 / kShare, kSets = kPeer ? 2 : 1;
    Iter it;
    Segment seg;
    int tile, end;
    int req, idx[kSets], tok[kSets], cnt, len, page[kSets];
    unsigned long long row[kSets];
    __device__ __forceinline__ void start(const Iter &from) { it = from; tile = end = 0; }
    __device__ __forceinline__ void open(const DecodeParams &p, int lane, int first) {
#pragma unroll
        for (int s = 0; s < kSets; ++s) row[s] = kSkip;
#pragma unroll 1
        for (int j = 0; j < kTiles; ++j) {
            if (tile == end) {
                if (!it.next(p, seg)) break;
                tile = seg.tile_begin; end = seg.tile_end;
            }
            if (lane / kShare == j) {
                const umma::TileGeom g = umma::tile_geom(seg.lo, seg.hi, tile * kPage);
                req = seg.request;
#pragma unroll
                for (int s = 0; s < kSets; ++s) {
                    const int r = (first + lane % kShare) ^ (s ? 32 : 0);
                    idx[s] = tile * kPage + g.tok0 + r;
                    row[s] = r >= g.r_lo && r < g.r_hi ? ~0ull : kSkip;          // (address to come)
                }
            }
            ++tile;
        }
    }
    __device__ __forceinline__ void link(const DecodeParams &p, int step) {
        bool any = row[0] != kSkip;
        if constexpr (kPeer) any |= row[1] != kSkip;
        if (!any) return;
        if (step == 0) { cnt = p.seq_lens[req]; len = p.ctx_lens[req]; }
#pragma unroll
        for (int s = 0; s < kSets; ++s) {
            if (row[s] == kSkip) continue;
            if (step == 0) {
                tok[s] = idx[s] < p.len_cap ? p.sel[(int64_t)req * p.sel_stride + idx[s]] : -1;
            } else if (step == 1) {
                // (a count outside [0, len_cap] stands for one poisoned row)
                if (cnt < 0 || cnt > p.len_cap || tok[s] >= len) tok[s] = -1;
                page[s] = tok[s] >= 0 ? p.block_table[(int64_t)req * p.table_stride + tok[s] / kPage] : -1;
            } else {
                row[s] = page[s] < 0 || page[s] >= p.num_pool_pages ? kPoison
                    : reinterpret_cast<unsigned long long>(p.kv_pool) + (unsigned long long)((int64_t)page[s] * kPage + tok[s] % kPage) * kSparseRowBytes;
            }
        }
    }
};

}  // namespace gather

// Warp gw of kGatherWarps: its rows of every tile of the worker.  kRows rows of a tile are this CTA's own (all 576 columns, for
// QK^T and P.V); of a pair, whose CTAs own 32 rows each, the two 128-column blocks of the OTHER 32 rows that this CTA multiplies
// follow two tiles later, into the chunk slots that QK^T has left (splash_decode_umma_pair.cu).
// stage(t): the first slab of tile t's stage.  wait_stage(t), wait_qk(t): it may be written, its other half's slots may.  Nothing here
// depends on whether a wait gave up: the warp walks its tiles to the end (no wait blocks once the CTA aborts), in step.  done_own(t), done_peer(t): all lanes, after their stores.
template <int kRows, typename Iter, typename Stage, typename WaitStage, typename DoneOwn, typename WaitQk, typename DonePeer>
__device__ __forceinline__ void gather_tiles(const DecodeParams &p, const Iter &it, int gw, int lane, int rank, Stage &&stage, WaitStage &&wait_stage,
                                             DoneOwn &&done_own, WaitQk &&wait_qk, DonePeer &&done_peer) {
    using namespace gather;
    constexpr bool kPeer = kRows == 32;
    constexpr int kShare = kRows / kGatherWarps;       // rows of a tile for this warp
    constexpr int kBatches = kShare / 4;               // four rows at a time
    constexpr uint32_t kSlabBytes = kRows * 128;
    constexpr int kLag = 2;
    Resolver<kShare, kPeer, Iter> res;
    res.start(it);
    const int batches = (it.end - it.x) * kBatches;
    if (batches == 0) return;
    const int first = (kPeer ? 32 * rank : 0) + gw * kShare;
    res.open(p, lane, first);
    for (int step = 0; step < 3; ++step) res.link(p, step);
    unsigned long long own = res.row[0], peer = kSkip, peer_before = kSkip;
    if constexpr (kPeer) peer = res.row[1];
    // a lane has 16 codes of each 128-code block, and 16 bytes of the rope part, of row lane / 8 of the four
    const int x = lane & 7;
    uint4 codes[4], rope, peer_codes[2];
    float4 scale;
    float peer_scale[2];
    auto load_scales = [](unsigned long long row) {
        const uint4 s = row > kPoison ? load_global16(row + kDLatent) : make_uint4(0x3f800000u, 0x3f800000u, 0x3f800000u, 0x3f800000u);
        return make_float4(__uint_as_float(s.x), __uint_as_float(s.y), __uint_as_float(s.z), __uint_as_float(s.w));
    };
    auto load_peer = [&](unsigned long long row) {
#pragma unroll
        for (int n = 0; n < 2; ++n) {
            peer_codes[n] = load16(row, (2 * n + rank) * 128 + 16 * x, kPoisonCodes);
            peer_scale[n] = 1.f;
            if (row > kPoison) asm volatile("ld.global.f32 %0, [%1];" : "=f"(peer_scale[n]) : "l"(row + kDLatent + (2 * n + rank) * 4) : "memory");
        }
    };
    {
        const unsigned long long row = __shfl_sync(0xffffffffu, own, lane >> 3);
#pragma unroll
        for (int j = 0; j < 4; ++j) codes[j] = load16(row, 128 * j + 16 * x, kPoisonCodes);
        scale = load_scales(row);
        rope = load16(row, kDLatent + 16 + 16 * x, kPoisonRope);
    }
    const int total = kPeer ? batches + kLag : batches;
#pragma unroll 1
    for (int i = 0; i < total; ++i) {
        const int k = i & 7;
        if (k == 0) {
            // the group that starts here was resolved during the one before it
            if (i > 0) {
                own = res.row[0];
                if constexpr (kPeer) { peer_before = peer; peer = res.row[1]; }
            }
            res.open(p, lane, first);
        } else if (k <= 3) {
            res.link(p, k - 1);
        }
        if (i < batches) {
            const uint32_t t = (uint32_t)i / kBatches;
            const int r = gw * kShare + (i % kBatches) * 4 + (lane >> 3);
            const unsigned long long next = __shfl_sync(0xffffffffu, k == 7 ? res.row[0] : own, ((k + 1) & 7) * 4 + (lane >> 3));
            if (i % kBatches == 0) wait_stage(t);
            uint8_t *const slab_row = stage(t) + r * 128;
            const float s[4] = {scale.x, scale.y, scale.z, scale.w};
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                dequant16(codes[j], s[j], slab_row + (2 * j + (x >> 2)) * kSlabBytes, r, 2 * (x & 3));
                codes[j] = load16(next, 128 * j + 16 * x, kPoisonCodes);
            }
            *reinterpret_cast<uint4 *>(slab_row + 8 * kSlabBytes + ((x ^ (r & 7)) << 4)) = rope;
            rope = load16(next, kDLatent + 16 + 16 * x, kPoisonRope);
            scale = load_scales(next);
            if (i % kBatches == kBatches - 1) done_own(t);
        }
        if constexpr (kPeer) {
            // the other half's rows of tile i - kLag, then the loads for the next one's (L2 hits, mostly: the peer reads them too)
            const int j = i - kLag;
            if (j >= 0) {
                wait_qk((uint32_t)j);
                const int r = gw * kShare + (lane >> 3);
                uint8_t *const slab_row = stage((uint32_t)j) + r * 128;
#pragma unroll
                for (int n = 0; n < 2; ++n)
                    dequant16(peer_codes[n], peer_scale[n], slab_row + (4 * n + 2 * (1 - rank) + (x >> 2)) * kSlabBytes, r, 2 * (x & 3));
                done_peer((uint32_t)j);
            }
            const int m = j + 1;                       // (in the group before this one while k < kLag - 1)
            if (m >= 0) load_peer(__shfl_sync(0xffffffffu, (m >> 3) == (i >> 3) ? peer : peer_before, (m & 7) * 4 + (lane >> 3)));
        }
    }
}

}  // namespace splash
