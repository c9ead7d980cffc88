// Shared declarations of the MLA decode library: dimensions, the split-KV work
// plan that the plan kernel writes into the caller's workspace, and host helpers.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>
#include <stddef.h>

#include <mutex>

#include "../../include/splash_mla.h"

namespace splash {

constexpr int kDQK = 576;        // d_c + d_r (absorbed MLA row width)
constexpr int kMaxQRows = 8;      // query rows per request (multi-token decode steps, short prefill chunks)
constexpr int kDV = 512;         // d_c (value width)
constexpr int kDRope = 64;
constexpr int kDLatent = 512;
constexpr int kPage = 64;        // tokens per page
constexpr int kMaxHeads = 128;
// largest page id (exclusive) the allocation-free migrate entry point can remap: 1 MiB of table
constexpr int kStaticMigrateMaxPageId = 1 << 18;

// Cost, in page tiles, charged once per non-empty request when the plan balances work
// over CTAs (query operands, pipeline refill, epilogue): measured per kernel, passed to the
// plan kernel at launch.
constexpr int kRequestOverheadTilesDefault = 4;
constexpr int kRequestOverheadTilesFp8 = 6;        // also right for the 16- / 32-head e4m3 kernel: a TP-8 share of the rollout
                                                   // workload takes 237 / 232 / 228 / 224 / 227 / 232 / 239 us with 2 / 3 / 4 / 6 / 8 / 10 / 14
constexpr int kRequestOverheadTilesPair = 5;       // bf16 CTA-pair kernel (a segment costs 7,500 cycles, a tile 1,650)
constexpr int kRequestOverheadTilesFp8Pair32 = 8;  // the same kernel with 32 heads per CTA
constexpr int kRequestOverheadTilesFp8Pair = 13;   // CTA-pair kernel: tiles are cheaper, the per-request work is not

// ---- workspace layout ------------------------------------------------------
// [0, 64)                 status block (int32 x 16): [0] status, [1..3] detail
// then int32 arrays       tile_start[B+1], req_lo[B], req_hi[B], req_wfirst[B],
//                         req_wlast[B], cost_start[B+1], worker_begin[W+1], split_list[W+1], worker_req[W+1]
//                         (status[8] = number of entries of split_list)
// then (16-B aligned)     split_rec [W+1] int4
// then (256-B aligned)    partial_lse [2W][h] fp32
// then (256-B aligned)    partial_scale [2W][h] fp32 (f16 partial outputs only: the power of two a row was divided by)
// then (256-B aligned)    partial_out [2W][h][512] fp32
struct PlanView {
    int32_t *status;        // 16 ints
    int32_t *tile_start;    // [B+1] exclusive prefix of per-request tile counts
    int32_t *req_lo;        // [B] first token of the effective range
    int32_t *req_hi;        // [B] one past the last token (>= lo; == lo when empty)
    int32_t *req_wfirst;    // [B] first worker holding a piece of the request (-1 if empty)
    int32_t *req_wlast;     // [B] last such worker
    int32_t *cost_start;    // [B+1] exclusive prefix of per-request cost (tiles + overhead)
    int32_t *worker_begin;  // [W+1] global tile index where each worker starts
    int32_t *split_list;    // [W+1] requests computed in more than one piece (count in status[8])
    int32_t *worker_req;    // [W+1] the request that holds a worker's first tile (what the kernels would bisect for)
    int4 *split_rec;        // [W+1] per entry of split_list: (request, first worker, last worker, SplitFlags)
    float *partial_lse;     // [2W][h]
    float *partial_scale;   // [2W][h]
    float *partial_out;     // [2W][h][512]
    int32_t num_workers;    // W
    int32_t h;              // width of the head slice
    size_t bytes;           // total bytes needed
};

inline __host__ __device__ size_t align_up(size_t x, size_t a) { return (x + a - 1) / a * a; }

inline __host__ PlanView make_plan_view(void *workspace, int B, int W, int h) {
    PlanView v;
    char *p = static_cast<char *>(workspace);
    size_t off = 0;
    v.status = reinterpret_cast<int32_t *>(p + off); off += 64;
    v.tile_start = reinterpret_cast<int32_t *>(p + off); off += sizeof(int32_t) * (size_t)(B + 1);
    v.req_lo = reinterpret_cast<int32_t *>(p + off); off += sizeof(int32_t) * (size_t)B;
    v.req_hi = reinterpret_cast<int32_t *>(p + off); off += sizeof(int32_t) * (size_t)B;
    v.req_wfirst = reinterpret_cast<int32_t *>(p + off); off += sizeof(int32_t) * (size_t)B;
    v.req_wlast = reinterpret_cast<int32_t *>(p + off); off += sizeof(int32_t) * (size_t)B;
    v.cost_start = reinterpret_cast<int32_t *>(p + off); off += sizeof(int32_t) * (size_t)(B + 1);
    v.worker_begin = reinterpret_cast<int32_t *>(p + off); off += sizeof(int32_t) * (size_t)(W + 1);
    v.split_list = reinterpret_cast<int32_t *>(p + off); off += sizeof(int32_t) * (size_t)(W + 1);
    v.worker_req = reinterpret_cast<int32_t *>(p + off); off += sizeof(int32_t) * (size_t)(W + 1);
    off = align_up(off, 16);
    v.split_rec = reinterpret_cast<int4 *>(p + off); off += sizeof(int4) * (size_t)(W + 1);
    off = align_up(off, 256);
    v.partial_lse = reinterpret_cast<float *>(p + off); off += sizeof(float) * (size_t)2 * W * h;
    off = align_up(off, 256);
    v.partial_scale = reinterpret_cast<float *>(p + off); off += sizeof(float) * (size_t)2 * W * h;
    off = align_up(off, 256);
    v.partial_out = reinterpret_cast<float *>(p + off); off += sizeof(float) * (size_t)2 * W * h * kDV;
    v.num_workers = W;
    v.h = h;
    v.bytes = off;
    return v;
}

// What a record says of a cut request's slots: a worker's piece lies in slot 2 w, the first worker's in 2 w + 1 if an earlier request's
// piece came before it.  Where all the work costs less than there are workers, the plan kernel lets several workers start on one tile, of
// which the last one has it: the cost stands above that bit then (else 0), and a combine kernel works out which they are.
enum SplitFlags { kSplitSecondSlot = 1, kSplitCostShift = 1 };

// Arguments common to the decode kernels.
struct DecodeParams {
    const void *q;
    const void *kv_pool;
    const float *kv_scales;
    const int32_t *block_table;
    const int32_t *seq_lens;
    float *out;
    float *lse;
    int64_t q_stride_request, q_stride_head;
    int64_t out_stride_request, out_stride_head;
    int64_t lse_stride_request;
    int32_t B, H;
    int32_t head_begin, head_end;
    int32_t table_stride;
    int32_t num_pool_pages;
    int32_t q_rows;            // R query rows per request; the heads of a call are then virtual heads g * R + r, and
                               // row r attends causally: tokens below seq_len - (R - 1 - r)
    int32_t heads_per_group;   // heads one CTA computes
    int32_t num_groups;        // head groups per KV worker
    int32_t pair_groups;       // CTA-pair kernels: CTA pairs per KV worker (1; more when several query rows per request
                               // make more than 128 (head, row) pairs: pair g of a worker takes pairs [128 g, 128 g + 128)
                               // and the pairs of a worker stream the same pages side by side, so the second read of a
                               // page hits L2 and the cache crosses HBM once)
    float softmax_scale;
    // plan (device pointers into the workspace)
    const int32_t *tile_start, *req_lo, *req_hi, *worker_begin;
    const int32_t *worker_req;   // request holding each worker's first tile, from the plan
    int32_t *status;
    float *partial_lse, *partial_out;
    float *partial_scale;      // f16 partial outputs: row (slot, head) holds O * 2^k with 2^-k stored here
    int32_t partial_f16;       // 1: the partial outputs are f16 (same slot order, rows of 512 halves): half the bytes for the
                               // decode kernel to write and the combine kernel to read; 11 significant bits of a normalised O,
                               // each row scaled by a power of two so that its largest entry sits just below f16's maximum
                               // (exact, and no limit on the magnitude of the cache values)
    int32_t len_cap;           // >= 0: seq_lens holds list counts; one outside [0, len_cap] counts as 1 (sparse decode)
    // sparse decode: kv_pool holds 656-byte rows, block_table / num_pool_pages describe it, and request i
    // attends over the tokens sel[i * sel_stride + j], j < seq_lens[i], each below ctx_lens[i]
    const int32_t *sel, *ctx_lens;
    int64_t sel_stride;
    int32_t sparse;
    int32_t num_workers;
    int32_t request_overhead_tiles;   // per-request cost the plan adds to the tile count
    int32_t plan_mode;                // kPlanWorkspace, kPlanInline or kPlanWhole
    int32_t q_by_hand;                // e4m3 pair kernel: its warps copy the query rows (strides that a tensor map cannot state)
    int32_t clear_status;             // 1: no plan kernel ran (its partition is taken again): block 0 clears the error words
    const int32_t *kv_begin, *kv_end; // the inline modes read the ranges themselves
    int4 *split_rec;                  // kPlanInline: where block 0 leaves the combine kernel's records
    long long *trace;          // optional device buffer for pipeline timestamps (diagnostics), or NULL
};

// A worker's next piece of work: request, its relative tile range, where the
// result goes.
struct Segment {
    int32_t request;
    int32_t tile_begin, tile_end;   // page-tile indices relative to floor(lo/64)
    int32_t lo, hi;                 // effective token range of the request
    int32_t slot;                   // partial slot, or -1 when the piece is the whole request
};

// ---- programmatic dependent launch ---------------------------------------------
// The three kernels of a decode call are chained with programmatic stream serialisation:
// a dependent kernel may be scheduled while its predecessor is still running, does its
// own set-up (barriers, tensor memory), and blocks in grid_dependency_wait() before it
// touches anything the predecessor wrote.
__device__ __forceinline__ void grid_dependency_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
// What a kernel reads behind its wait may have been written while it was already resident, by the kernel in front of it.  So it is
// never read through the read-only path (__ldg, const __restrict__ parameters): such data counts as unchanged for the kernel's
// lifetime, and a load of it may be moved over the wait.  Plain loads may not; nor these, which go to L2 past a line that a read
// before the wait has left in L1, and are not merged with that read.
__device__ __forceinline__ int32_t load_l2(const int32_t *ptr) {
    int32_t v;
    asm volatile("ld.global.cg.b32 %0, [%1];" : "=r"(v) : "l"(ptr) : "memory");
    return v;
}
__device__ __forceinline__ void grid_launch_dependents() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }

// Where a decode kernel's partition comes from.  Workspace: the plan kernel wrote it.  Inline: a batch of at most 32
// requests is one lane each, so a warp of every CTA works the partition out for itself in a shuffle scan while the plan
// kernel of such a call would still be in its launch (a tiny decode: 16.4 us with the plan kernel in front, see
// build_inline_plan); the requests are cut where the plan kernel cuts them, though by other workers where all the work costs less than
// there are (cut_workers).  Whole: inline, and no request is cut -- worker i takes request
// i -- so that there is nothing to combine either.
enum { kPlanWorkspace = 0, kPlanInline = 1, kPlanWhole = 2 };
constexpr int kInlinePlanRequests = 32;
// (contexts of at most this many pages: 4 requests in a table as wide as they are against one of 2,048 columns, whose requests are cut and
// combined: 16 heads 11.9 against 15 to 16 us, 128 heads 11.1 against 13.8, e4m3 9.1 against 12.8 and 16.9 against 21.4)
constexpr int kWholeRequestPages = 4;
// shared-memory copy of an inline plan: tile_start[B + 1], lo[B], hi[B] (as in the workspace), then the worker's first
// tile, its end, and the request that holds the first
constexpr uint32_t kInlinePlanBytes = ((3 * kInlinePlanRequests + 4) * 4 + 15) / 16 * 16;

// Effective range of request i (the rule of the plan kernel).
__device__ __forceinline__ void effective_range(int s, const int32_t *kv_begin, const int32_t *kv_end, int i, int len_cap, int &lo, int &hi) {
    if (len_cap >= 0 && (s < 0 || s > len_cap)) s = 1;     // a list count out of bounds: one (poisoned) row
    lo = kv_begin ? load_l2(kv_begin + i) : 0;
    hi = kv_end ? load_l2(kv_end + i) : s;
    if (lo < 0) lo = 0;
    if (hi > s) hi = s;
    if (hi < lo) hi = lo;
}

// floor(total * w / W) without 64-bit division: total = a W + b, floor = a w + floor(b w / W)
__device__ __forceinline__ int cost_target(int total, int w, int W) {
    const int a = total / W, b = total - a * W;
    return a * w + (b * w) / W;
}

// The lengths of a batch of at most 32 requests, a request per lane: its effective range.
__device__ __forceinline__ void lane_range(const DecodeParams &p, int lane, int &lo, int &hi) {
    lo = hi = 0;
    if (lane < p.B) effective_range(load_l2(p.seq_lens + lane), p.kv_begin, p.kv_end, lane, p.len_cap, lo, hi);
}

// Workers that an inline plan cuts the work for: no more than the work costs (tiles, and the overhead of each request).  Their shares
// then begin at different costs, so that from the first to the last worker of a request each has a piece of it, as the combine kernel takes
// for granted.  (A worker whose share begins in a request's overhead, where the next one's does too, has nothing: it stands in front of
// that request's first worker.)
__device__ __forceinline__ int cut_workers(const DecodeParams &p, int cost) { return min(p.num_workers, cost); }

// One warp of a CTA: the plan, as far as worker `worker` needs it, from the lanes' ranges.
static __device__ __noinline__ void build_inline_plan(const DecodeParams &p, int worker, int32_t *sp, int lane, int lo, int hi) {
    const int B = p.B, overhead = p.request_overhead_tiles;
    const int n = hi > lo ? (hi + kPage - 1) / kPage - lo / kPage : 0;
    const int c = n > 0 ? n + overhead : 0;
    int sn = n, sc = c;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int a = __shfl_up_sync(0xffffffffu, sn, o), b = __shfl_up_sync(0xffffffffu, sc, o);
        if (lane >= o) { sn += a; sc += b; }
    }
    if (lane == 0) sp[0] = 0;
    if (lane < B) { sp[lane + 1] = sn; sp[B + 1 + lane] = lo; sp[2 * B + 1 + lane] = hi; }
    if (p.plan_mode == kPlanWhole) {
        if (lane == worker) { sp[3 * B + 1] = sn - n; sp[3 * B + 2] = sn; sp[3 * B + 3] = worker; }
        return;
    }
    const int tiles = __shfl_sync(0xffffffffu, sn, 31), cost = __shfl_sync(0xffffffffu, sc, 31), W = cut_workers(p, cost);
    // first tile of worker w (the same w in all lanes) and the request that holds it: as many requests lie before it as
    // end at or before its share of the cost
    auto start = [&](int w, int &req) {
        req = 0;
        if (w >= W) return tiles;
        const int target = cost_target(cost, w, W);
        req = __popc(__ballot_sync(0xffffffffu, sc <= target));
        const int off = target - __shfl_sync(0xffffffffu, sc - c, req) - overhead;
        return __shfl_sync(0xffffffffu, sn - n, req) + max(off, 0);
    };
    int req, unused;
    const int wb = start(worker, req), we = start(worker + 1, unused);
    if (lane == 0) { sp[3 * B + 1] = wb; sp[3 * B + 2] = we; sp[3 * B + 3] = req; }
}

// What of the cache a CTA loads first: `bytes` at `offset` of the pages of the worker's first `count` tiles; and its heads.
struct FirstLoads { uint32_t page_bytes, offset, bytes; int count, head0, heads; };

// Before grid_dependency_wait, the same warp: the plan from the lengths as they lie there now, and from it the worker's first
// pages, their scales and its first request's query rows into L2, while the work before this call on the stream still
// runs (in a loop over layers the combine kernel of the one before: microseconds in which DRAM is idle).  Nothing of this is
// relied on: the lengths are read again after the wait, and the plan made again if they differ; what is prefetched is
// only that.  All reads go to L2 (a line in L1 would be stale after the wait).
static __device__ __noinline__ void plan_ahead(const DecodeParams &p, int worker, int32_t *sp, int lane, const FirstLoads &f, int &lo, int &hi) {
    lane_range(p, lane, lo, hi);
    build_inline_plan(p, worker, sp, lane, lo, hi);
    __syncwarp();
    const int B = p.B, wb = sp[3 * B + 1], we = sp[3 * B + 2], req = sp[3 * B + 3];
    if (wb < 0 || wb >= we || req < 0 || req >= B) return;
    const int x = wb + lane;
    if (!p.sparse && lane < f.count && x < we) {
        int r = req;
        while (r + 1 < B && sp[r + 1] <= x) ++r;
        const int64_t idx = (int64_t)sp[B + 1 + r] / kPage + (x - sp[r]);
        if (idx >= 0 && idx < p.table_stride) {
            const int page = load_l2(p.block_table + (int64_t)r * p.table_stride + idx);
            if (page >= 0 && page < p.num_pool_pages) {
                asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;"
                             ::"l"(static_cast<const uint8_t *>(p.kv_pool) + (size_t)page * f.page_bytes + f.offset), "r"(f.bytes) : "memory");
                if (p.kv_scales != nullptr) {
                    asm volatile("prefetch.global.L2 [%0];" ::"l"(p.kv_scales + (size_t)page * kPage));
                    asm volatile("prefetch.global.L2 [%0];" ::"l"(p.kv_scales + (size_t)page * kPage + 32));
                }
            }
        }
    }
    const char *q = static_cast<const char *>(p.q) + ((int64_t)req * p.q_stride_request + (int64_t)f.head0 * p.q_stride_head) * 2;
    const int rows = min(f.heads, p.head_end - f.head0);
    for (int i = lane; i < rows * 9; i += 32) asm volatile("prefetch.global.L2 [%0];" ::"l"(q + (int64_t)(i / 9) * p.q_stride_head * 2 + (i % 9) * 128));
}

// What the combine kernel reads: the plan's warp of block 0 leaves the list of the requests that were cut, once its CTA is under way, and clears
// the status block (this cannot wipe another CTA's report: the first
// one a CTA can make is the end of a bounded wait, seconds after this).  A lane knows the first and the last worker of its request
// from the costs alone: worker w starts at or before tile t of a request whose cost begins at c iff floor(w cost / W) <= c + overhead + t,
// so the last such worker is floor(((c + overhead + t + 1) W - 1) / cost).  (Block 0 going through all workers for every request was
// late by microseconds at many requests: 32 of 2,048 tokens, 16 heads over e4m3, 23.7 us a call, now 20.2.)
static __device__ __noinline__ void publish_inline_plan(const DecodeParams &p, const int32_t *ts, int lane) {
    const int B = p.B, overhead = p.request_overhead_tiles;
    int split = 0;
    if (p.plan_mode == kPlanInline) {
        const int n = lane < B ? ts[lane + 1] - ts[lane] : 0;
        int sc = n > 0 ? n + overhead : 0;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int b = __shfl_up_sync(0xffffffffu, sc, o);
            if (lane >= o) sc += b;
        }
        const int cost = __shfl_sync(0xffffffffu, sc, 31), W = cut_workers(p, cost);
        int wf = 0, wl = 0;
        if (n > 0) {
            auto worker_before = [&](int c) { return min(W - 1, (int)(((unsigned long long)(unsigned)c * (unsigned)W - 1) / (unsigned)cost)); };
            wf = worker_before(sc - n + 1);        // (the cost up to and with the first tile, and with the last)
            wl = worker_before(sc);
        }
        const unsigned cut = __ballot_sync(0xffffffffu, wf != wl);
        split = __popc(cut);
        if ((cut >> lane) & 1u) p.split_rec[__popc(cut & ((1u << lane) - 1u))] = make_int4(lane, wf, wl, (long long)wf * cost < (long long)(sc - n - overhead) * W ? kSplitSecondSlot : 0);      // (its share starts in front of the request's)
    }
    if (lane < 16) p.status[lane] = lane == 8 ? split : 0;
}

// Iterates the segments of worker w in plan order.  Every thread of a CTA calls
// it with the same arguments and gets the same answer.  kPlanOffset: where an inline plan lies in dynamic shared memory;
// kPlanInWorkspace: the kernel is launched behind a plan kernel only.
constexpr uint32_t kPlanInWorkspace = 0xffffffffu;
template <uint32_t kPlanOffset>
struct SegmentIter {
    int32_t x, end, wb, i, w;
    static __device__ __forceinline__ int32_t *inline_plan() {
        extern __shared__ __align__(1024) uint8_t smem[];
        return reinterpret_cast<int32_t *>(smem + kPlanOffset);
    }
    // tile_start[B + 1]; lo[B] and hi[B] follow it, in the workspace and in an inline plan alike
    static __device__ __forceinline__ const int32_t *tile_start(const DecodeParams &p) {
        return p.plan_mode != kPlanWorkspace ? inline_plan() : p.tile_start;
    }
    __device__ void init(const DecodeParams &p, int worker) {
        w = worker;
        // i: the request containing tile x (last i with ts[i] <= x and ts[i+1] > x): the plan has it, which saves every
        // role of every CTA a bisection of a dozen dependent global loads before its first tile
        if (p.plan_mode != kPlanWorkspace) {
            const int32_t *own = inline_plan() + 3 * p.B + 1;
            wb = own[0]; x = wb; end = own[1]; i = own[2];
        } else {
            wb = p.worker_begin[worker]; x = wb; end = p.worker_begin[worker + 1];
            i = x < end ? p.worker_req[worker] : 0;
        }
    }
    __device__ bool next(const DecodeParams &p, Segment &s) {
        if (x >= end) return false;
        const int32_t *ts = tile_start(p);
        while (ts[i + 1] <= x) ++i;                    // skip finished / empty requests
        int rs = ts[i], re = ts[i + 1];
        int seg_end = re < end ? re : end;
        s.request = i;
        s.tile_begin = x - rs;
        s.tile_end = seg_end - rs;
        s.lo = ts[p.B + 1 + i];
        s.hi = ts[2 * p.B + 1 + i];
        bool full = (x == rs) && (seg_end == re);
        s.slot = full ? -1 : 2 * w + (rs <= wb ? 0 : 1);
        x = seg_end;
        return true;
    }
};

// The same on the workspace's arrays only.
template <>
struct SegmentIter<kPlanInWorkspace> {
    const int32_t *ts;
    int32_t B, x, end, wb, i, w;
    static __device__ __forceinline__ const int32_t *tile_start(const DecodeParams &p) { return p.tile_start; }
    __device__ void init(const DecodeParams &p, int worker) {
        ts = p.tile_start; B = p.B; w = worker;
        wb = p.worker_begin[worker]; x = wb; end = p.worker_begin[worker + 1];
        i = x < end ? p.worker_req[worker] : 0;
    }
    __device__ bool next(const DecodeParams &p, Segment &s) {
        if (x >= end) return false;
        while (ts[i + 1] <= x) ++i;
        int rs = ts[i], re = ts[i + 1];
        int seg_end = re < end ? re : end;
        s.request = i;
        s.tile_begin = x - rs;
        s.tile_end = seg_end - rs;
        s.lo = p.req_lo[i];
        s.hi = p.req_hi[i];
        bool full = (x == rs) && (seg_end == re);
        s.slot = full ? -1 : 2 * w + (rs <= wb ? 0 : 1);
        x = seg_end;
        return true;
    }
};

// The beginning of a decode kernel, all threads, around its grid_dependency_wait: the plan's origin by the call's mode.
// `plan_warp`: a warp that is not needed at once.  kAhead: the kernel leaves a combine block room beside its CTA, so its CTAs are
// there well before the wait ends and may plan ahead; where they come in only as the blocks before them leave, planning twice
// is time lost (1 us of a call).  A call that cuts no request has no combine kernel in front of the next one: always ahead.
template <bool kAhead, uint32_t kPlanOffset>
__device__ __forceinline__ void start_plan(const DecodeParams &p, int worker, int plan_warp, SegmentIter<kPlanOffset> &it, const FirstLoads &f) {
    if constexpr (kPlanOffset != kPlanInWorkspace) {
        if (p.plan_mode != kPlanWorkspace) {
            const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
            int32_t *sp = it.inline_plan();
            int lo = 0, hi = 0;
            const bool ahead = kAhead || p.plan_mode == kPlanWhole;
            if (ahead && warp == plan_warp) plan_ahead(p, worker, sp, lane, f, lo, hi);
            grid_dependency_wait();
            // no combine kernel follows and every CTA is running: the next call's first kernel may set up on the SMs left
            if (p.plan_mode == kPlanWhole) grid_launch_dependents();
            if (warp == plan_warp) {
                int lo2, hi2;
                lane_range(p, lane, lo2, hi2);
                if (!ahead || __any_sync(0xffffffffu, lo2 != lo || hi2 != hi)) build_inline_plan(p, worker, sp, lane, lo2, hi2);
            }
            __syncthreads();
            if (blockIdx.x == 0 && warp == plan_warp) publish_inline_plan(p, sp, lane);
            it.init(p, worker);
            return;
        }
    }
    grid_dependency_wait();       // the plan kernel's output is read from here on
    if (p.clear_status && blockIdx.x == 0 && threadIdx.x < 8) p.status[threadIdx.x] = 0;      // (see publish_inline_plan)
    it.init(p, worker);
}

// Requests whose effective KV range is empty belong to no segment: O = 0, LSE = -inf is
// written by the decode CTA (worker, head group) with worker == request mod num_workers,
// for its own heads.  Called by all threads of the CTA once its segments are done.
// `ts`: the plan's tile_start (SegmentIter::ts).
__device__ __forceinline__ void fill_empty_requests(const DecodeParams &p, const int32_t *ts, int worker, int head0, int heads_per_group,
                                                    int tid, int nthreads) {
    // The plan's arrays are a launch old and have left the caches: a loop over this worker's requests that looks at one
    // request per iteration is a chain of round trips to DRAM at the very end of the CTA (seven on the rollout workload).
    // Instead every lane looks at a request of its own -- one round trip -- and the warp then zeroes what it found.
    const int nheads = min(heads_per_group, p.head_end - head0);
    const int lane = tid & 31, wid = tid >> 5, nwarps = nthreads >> 5;
    for (int64_t j0 = (int64_t)wid * 32; worker + j0 * p.num_workers < p.B; j0 += (int64_t)nwarps * 32) {
        const int64_t mine = worker + (j0 + lane) * p.num_workers;
        const bool empty = mine < p.B && ts[mine + 1] == ts[mine];
        unsigned found = __ballot_sync(0xffffffffu, empty);
        while (found) {
            const int src = __ffs(found) - 1;
            found &= found - 1;
            const int64_t i = worker + (j0 + src) * p.num_workers;
            for (int idx = lane; idx < nheads * (kDV / 4); idx += 32) {
                const int hh = idx / (kDV / 4), c = idx % (kDV / 4);
                reinterpret_cast<float4 *>(p.out + i * p.out_stride_request + (int64_t)(head0 + hh) * p.out_stride_head)[c] =
                    make_float4(0.f, 0.f, 0.f, 0.f);
            }
            for (int hh = lane; hh < nheads; hh += 32) p.lse[i * p.lse_stride_request + head0 + hh] = -INFINITY;
        }
    }
}

template <typename... KArgs, typename... Args>
inline cudaError_t launch_dependent(void (*kernel)(KArgs...), dim3 grid, dim3 block, size_t smem, cudaStream_t stream,
                                    Args &&...args) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid; cfg.blockDim = block; cfg.dynamicSmemBytes = smem; cfg.stream = stream;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr; cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, kernel, static_cast<KArgs>(args)...);
}

// Per-device one-time set-up of a launcher (function attributes are per device).  The set-up runs under a lock and a
// device counts as done only once it has succeeded, so a second host thread whose first call on a device comes at the
// same time waits for the attribute to be in place instead of launching without it.
struct DeviceOnce {
    std::mutex mu;
    bool done[64] = {};
    template <typename F>
    cudaError_t run(F &&setup) {
        int dev = 0;
        if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return setup();
        std::lock_guard<std::mutex> lock(mu);
        if (done[dev]) return cudaSuccess;
        const cudaError_t e = setup();
        if (e == cudaSuccess) done[dev] = true;
        return e;
    }
};

// ---- host helpers (splash_api.cu) -----------------------------------------
void set_error(const char *fmt, ...);
void count_launch(int n = 1);

// kernels' host launchers
cudaError_t launch_plan(const DecodeParams &p, const PlanView &v, cudaStream_t stream);
cudaError_t launch_validate_pages(const DecodeParams &p, const int32_t *req_lo, const int32_t *req_hi, cudaStream_t stream);
cudaError_t launch_sparse_gather(int B, int max_sel, int pages_per_request, const void *kv_pool, int num_pool_pages,
                                 const int32_t *block_table, int64_t table_stride, const int32_t *seq_lens,
                                 const int32_t *sel, int64_t sel_stride, const int32_t *sel_count, void *dense_pool,
                                 int32_t *dense_table, int sm_count, cudaStream_t stream);
cudaError_t launch_dop_pack_rows(const void *a, const void *b, void *out, const int32_t *send_row, int64_t n, int h,
                                 int64_t a_bytes, int64_t b_bytes, int64_t a_row_pitch, int64_t a_head_pitch,
                                 int64_t b_row_pitch, int64_t b_head_pitch, int sm_count, cudaStream_t stream);
cudaError_t launch_dop_unpack_rows(const void *recv, void *out, const int32_t *send_row, int64_t n, int64_t row_bytes,
                                   int64_t out_row_pitch, int sm_count, cudaStream_t stream);
cudaError_t launch_dop_swap_outer(const void *in, void *out, int64_t A, int64_t Bn, int64_t inner_bytes, int sm_count, cudaStream_t stream);
cudaError_t launch_decode_simt(const DecodeParams &p, int kv_dtype, cudaStream_t stream);
int simt_heads_per_group();
// tcgen05 kernel: how it cuts a head slice of width h into CTAs, and its launcher
void umma_tiling(int kv_dtype, int h, int sm_count, bool pairs, int *heads_per_group, int *num_groups, int *num_workers);
cudaError_t launch_decode_umma(const DecodeParams &p, const splash_mla_shape &shape, cudaStream_t stream);
cudaError_t launch_decode_umma_fp8(const DecodeParams &p, cudaStream_t stream);
cudaError_t launch_decode_umma_fp8_narrow(const DecodeParams &p, cudaStream_t stream);   // 16 / 32 heads per CTA
cudaError_t launch_decode_umma_fp8_pair(const DecodeParams &p, cudaStream_t stream);
cudaError_t launch_decode_umma_pair(const DecodeParams &p, cudaStream_t stream);
cudaError_t launch_split_combine(const DecodeParams &p, const int4 *split_rec, int sm_count, cudaStream_t stream);
cudaError_t launch_lse_merge(int num_parts, int64_t rows, int d_v, const float *part_out,
                             const float *part_lse, float *out, float *lse, int sm_count, cudaStream_t stream);
cudaError_t launch_page_migrate(const void *src_pool, const float *src_scales, void *dst_pool,
                                float *dst_scales, int64_t page_bytes, const int32_t *src_ids,
                                const int32_t *dst_ids, int64_t n, int32_t src_base, int32_t dst_base,
                                int32_t max_page_id, int32_t *block_table, int64_t num_entries,
                                int32_t *remap, int sm_count, cudaStream_t stream);

cudaError_t static_remap_address(int32_t **ptr);

}  // namespace splash
