// Split-KV work plan (device side, integer only, deterministic).
//
// The attention time of a decode step is set by the KV bytes read and the
// contraction work, both linear in the context length (the paper's per-step cost
// model, App. B: t_att = max{F_att / Phi_att, K_read / beta_KV}), so the plan
// spreads page tiles -- not requests -- evenly over the CTAs: the global sequence of
// (request, page tile) pairs is cut into `num_workers` contiguous runs of equal cost,
// where a non-empty request costs its tile count plus a fixed overhead.  A run that
// covers a whole request writes the final result; the (at most two) partial pieces
// at the ends of a run go to per-worker partial slots and are combined afterwards.
// The plan depends only on (seq_lens, kv ranges, shape), so a repeated call takes
// the same split and is bit-reproducible.
#include "splash_common.cuh"

namespace splash {

namespace {

constexpr int kPlanThreads = 1024;
constexpr int kPlanSmemRequests = 4096;
constexpr int kPlanSmemWorkers = 512;

// One CTA between the caller's work and the decode kernel: its time is latency (a load of the lengths, a scan, two
// bisections, the stores) and comes on top of every call of more than 32 requests.  As many threads as there are requests
// or workers, one barrier per 1,024 requests in the scan, 32-bit arithmetic.
__global__ void __launch_bounds__(kPlanThreads)
plan_kernel(int B, int W, int overhead, int len_cap, const int32_t *seq_lens, const int32_t *kv_begin,
            const int32_t *kv_end, int32_t *tile_start,
            int32_t *__restrict__ req_lo, int32_t *__restrict__ req_hi,
            int32_t *__restrict__ req_wfirst, int32_t *__restrict__ req_wlast,
            int32_t *cost_start, int32_t *worker_begin, int32_t *__restrict__ split_list, int32_t *__restrict__ worker_req,
            int4 *__restrict__ split_rec, int32_t *__restrict__ status) {
    __shared__ int2 warp_tot[2][32];
    __shared__ int n_split;
    // The bisections below chase a dozen dependent loads each; for the usual sizes the
    // prefix arrays live in shared memory while the plan is built and are copied out at the end.
    __shared__ int32_t s_tile[kPlanSmemRequests + 1], s_cost[kPlanSmemRequests + 1], s_wbeg[kPlanSmemWorkers + 1];
    const bool staged = B <= kPlanSmemRequests && W <= kPlanSmemWorkers;
    int32_t *const g_tile_start = tile_start, *const g_cost_start = cost_start, *const g_worker_begin = worker_begin;
    if (staged) { tile_start = s_tile; cost_start = s_cost; worker_begin = s_wbeg; }
    const int tid = threadIdx.x, nthreads = blockDim.x, lane = tid & 31, wid = tid >> 5;
    grid_dependency_wait();       // launched while the work before it on the stream still runs
    grid_launch_dependents();     // the next kernel may start its set-up now; it waits for this grid before reading the plan
    if (tid < 16) status[tid] = 0;
    if (tid == 0) { tile_start[0] = 0; cost_start[0] = 0; n_split = 0; }

    // pass 1: effective ranges, tile counts, exclusive prefixes of tiles and of cost
    int carry_tiles = 0, carry_cost = 0;
    for (int base = 0, chunk = 0; base < B; base += nthreads, ++chunk) {
        const int i = base + tid;
        int n = 0;
        if (i < B) {
            int lo, hi;
            effective_range(seq_lens[i], kv_begin, kv_end, i, len_cap, lo, hi);
            req_lo[i] = lo; req_hi[i] = hi;
            if (hi > lo) n = (hi + kPage - 1) / kPage - lo / kPage;
        }
        int sn = n, sc = n > 0 ? n + overhead : 0;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int a = __shfl_up_sync(0xffffffffu, sn, o), b = __shfl_up_sync(0xffffffffu, sc, o);
            if (lane >= o) { sn += a; sc += b; }
        }
        if (lane == 31) warp_tot[chunk & 1][wid] = make_int2(sn, sc);
        __syncthreads();
        // every warp scans the warps' totals for itself (two buffers: one barrier per chunk is enough)
        int2 t = lane < (nthreads >> 5) ? warp_tot[chunk & 1][lane] : make_int2(0, 0);
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int a = __shfl_up_sync(0xffffffffu, t.x, o), b = __shfl_up_sync(0xffffffffu, t.y, o);
            if (lane >= o) { t.x += a; t.y += b; }
        }
        const int before_n = wid > 0 ? __shfl_sync(0xffffffffu, t.x, (wid + 31) & 31) : 0;
        const int before_c = wid > 0 ? __shfl_sync(0xffffffffu, t.y, (wid + 31) & 31) : 0;
        if (i < B) { tile_start[i + 1] = carry_tiles + before_n + sn; cost_start[i + 1] = carry_cost + before_c + sc; }
        carry_tiles += __shfl_sync(0xffffffffu, t.x, 31);
        carry_cost += __shfl_sync(0xffffffffu, t.y, 31);
    }
    const int total_cost = carry_cost, total_tiles = carry_tiles;
    __threadfence_block();
    __syncthreads();

    // pass 2: worker w starts at cost floor(w * total_cost / W); the request whose
    // cost interval [cost_start[i], cost_start[i+1]) holds that value is found by
    // bisection, and a start that falls into the request's fixed overhead snaps to
    // its first tile.
    for (int w = tid; w <= W; w += nthreads) {
        int g = total_tiles, first_req = 0;
        if (w < W && total_cost > 0) {
            const int target = cost_target(total_cost, w, W);
            int lo = 0, hi = B;   // invariant cost_start[lo] <= target < cost_start[hi]
            while (hi - lo > 1) { int mid = (lo + hi) >> 1; if (cost_start[mid] <= target) lo = mid; else hi = mid; }
            while (cost_start[lo + 1] <= target) ++lo;   // (defensive; bisection already lands on a non-empty request)
            const int off = target - cost_start[lo] - overhead;
            g = tile_start[lo] + max(off, 0);
            first_req = lo;
        }
        worker_begin[w] = g;
        worker_req[w] = first_req;
    }
    __threadfence_block();
    __syncthreads();

    // pass 3: first / last worker of every request
    for (int i = tid; i < B; i += nthreads) {
        const int rs = tile_start[i], re = tile_start[i + 1];
        int wf = -1, wl = -1;
        if (re > rs) {
            // worker containing tile x: the w with worker_begin[w] <= x < worker_begin[w+1]; both bisections side by side
            int hi0 = W, hi1 = W;
            wf = wl = 0;          // invariant worker_begin[w] <= x < worker_begin[hi]
            while (hi0 - wf > 1 || hi1 - wl > 1) {
                const int m0 = (wf + hi0) >> 1, m1 = (wl + hi1) >> 1;
                const int b0 = worker_begin[m0], b1 = worker_begin[m1];
                if (hi0 - wf > 1) { if (b0 <= rs) wf = m0; else hi0 = m0; }
                if (hi1 - wl > 1) { if (b1 <= re - 1) wl = m1; else hi1 = m1; }
            }
        }
        req_wfirst[i] = wf; req_wlast[i] = wl;
        // requests cut into several pieces are listed for the combine kernel (at most W - 1 of them;
        // the list order varies from run to run, the results do not depend on it)
        if (wf != wl) {
            const int e = atomicAdd(&n_split, 1);
            split_list[e] = i;
            // all the combine kernel needs to know about the request, in one load
            split_rec[e] = make_int4(i, wf, wl, (worker_begin[wf] < rs ? kSplitSecondSlot : 0) | (total_cost < W ? total_cost << kSplitCostShift : 0));
        }
    }
    if (staged) {
        for (int i = tid; i <= B; i += nthreads) { g_tile_start[i] = s_tile[i]; g_cost_start[i] = s_cost[i]; }
        for (int w = tid; w <= W; w += nthreads) g_worker_begin[w] = s_wbeg[w];
    }
    __syncthreads();
    if (tid == 0) status[8] = n_split;
}

// Validation mode: every block-table entry of a page that intersects a request's effective range must name a page of
// the pool.  One block per request (grid-stride), threads over its pages; the first offender found wins the status word.
__global__ void __launch_bounds__(256)
validate_pages_kernel(int B, int num_pool_pages, int table_stride, const int32_t *__restrict__ block_table,
                      const int32_t *__restrict__ req_lo, const int32_t *__restrict__ req_hi, int32_t *status) {
    for (int i = blockIdx.x; i < B; i += gridDim.x) {
        const int lo = req_lo[i], hi = req_hi[i];
        if (hi <= lo) continue;
        for (int pg = lo / kPage + threadIdx.x; pg < (hi + kPage - 1) / kPage; pg += blockDim.x) {
            const int id = block_table[(int64_t)i * table_stride + pg];
            if (id < 0 || id >= num_pool_pages) {
                if (atomicCAS(status, 0, (int)SPLASH_BAD_PAGE_ID) == 0) { status[1] = i; status[2] = pg; status[3] = id; }
            }
        }
    }
}

}  // namespace

cudaError_t launch_validate_pages(const DecodeParams &p, const int32_t *req_lo, const int32_t *req_hi, cudaStream_t stream) {
    const int grid = p.B < 1024 ? p.B : 1024;
    validate_pages_kernel<<<grid, 256, 0, stream>>>(p.B, p.num_pool_pages, p.table_stride, p.block_table, req_lo, req_hi, p.status);
    count_launch();
    return cudaGetLastError();
}

cudaError_t launch_plan(const DecodeParams &p, const PlanView &v, cudaStream_t stream) {
    // same shared-memory carve-out as the decode kernel that follows: no reconfiguration between them
    static DeviceOnce once;
    once.run([&] {
        cudaFuncSetAttribute(plan_kernel, cudaFuncAttributePreferredSharedMemoryCarveout, cudaSharedmemCarveoutMaxShared);
        return cudaSuccess;     // a preference: a failure is not an error
    });
    const int items = p.B > p.num_workers + 1 ? p.B : p.num_workers + 1;
    const int threads = items >= kPlanThreads ? kPlanThreads : (items + 31) / 32 * 32;
    const cudaError_t e = launch_dependent(plan_kernel, dim3(1), dim3(threads), 0, stream, p.B, p.num_workers, p.request_overhead_tiles,
                                           p.len_cap, p.seq_lens, p.kv_begin, p.kv_end, v.tile_start, v.req_lo, v.req_hi, v.req_wfirst,
                                           v.req_wlast, v.cost_start, v.worker_begin, v.split_list, v.worker_req, v.split_rec, v.status);
    count_launch();
    return e;
}

}  // namespace splash
