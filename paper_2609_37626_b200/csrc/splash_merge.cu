// Log-sum-exp merges: the public CP merge (splash_lse_merge) and the reduction of
// the decode kernels' split-KV partial slots.  Both compute, per row,
//     L = ln sum_j exp(L_j),   O = sum_j exp(L_j - L) O_j,
// parts with L_j = -inf contributing nothing.  Pure fp32, HBM-bound.
#include <cuda_fp16.h>

#include <type_traits>

#include "splash_common.cuh"

namespace splash {

namespace {

constexpr int kMergeThreads = 128;

// What the LSEs of a row are measured against: their largest, or 0 where that is -inf.  Either no part saw a token then, and the
// weights add up to exactly 0, or an LSE is NaN (which fmaxf passes over), and so is the sum: the row becomes NaN, not empty.
__device__ __forceinline__ float reference_max(float m) { return m == -INFINITY ? 0.f : m; }

// One CTA per row and 128 float4 columns, a column per thread, where the rows are few (launch_lse_merge).  (A CTA that goes over all columns of a
// wide row has too few loads in flight then: 64 rows of four parts, 8,192 wide, 11.5 us, now 3.8.)  The parts' LSEs come in one load each, a part per
// thread, and the parts' rows kDepth loads at a time: taken one after the other in every thread they were a chain of round trips
// (128 rows of eight parts: 3.0 us, now 2.6; 24,960 of five: 77.5, now 55.4).  Where the rows are more
// than the SMs hold at a time, four loads each and twelve blocks to an SM instead of eight.
template <int kDepth>
__global__ void __launch_bounds__(kMergeThreads, kDepth == 8 ? 8 : 12)
lse_merge_kernel(int num_parts, int64_t rows, int d_v, const float *part_out, const float *part_lse, float *out, float *lse) {
    __shared__ float w_s[kMergeThreads], red_s[2][kMergeThreads / 32];
    grid_launch_dependents();
    grid_dependency_wait();       // launched while the work before it on the stream still runs
    const int64_t r = blockIdx.x;
    const int tid = threadIdx.x;
    float4 *o4 = reinterpret_cast<float4 *>(out + r * d_v);
    const int nvec = d_v / 4, c_first = blockIdx.y * kMergeThreads + tid, c_step = gridDim.y * kMergeThreads;
    const float first = tid < num_parts ? part_lse[(int64_t)tid * rows + r] : -INFINITY;
    float m = first;
    for (int j = tid + kMergeThreads; j < num_parts; j += kMergeThreads) m = fmaxf(m, part_lse[(int64_t)j * rows + r]);
    for (int o = 16; o; o >>= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, o));
    if ((tid & 31) == 0) red_s[0][tid >> 5] = m;
    __syncthreads();
    m = reference_max(fmaxf(fmaxf(red_s[0][0], red_s[0][1]), fmaxf(red_s[0][2], red_s[0][3])));
    float Z = expf(first - m);        // (0 for a part without tokens)
    for (int j = tid + kMergeThreads; j < num_parts; j += kMergeThreads) Z += expf(part_lse[(int64_t)j * rows + r] - m);
    for (int o = 16; o; o >>= 1) Z += __shfl_xor_sync(0xffffffffu, Z, o);
    if ((tid & 31) == 0) red_s[1][tid >> 5] = Z;
    __syncthreads();
    Z = (red_s[1][0] + red_s[1][1]) + (red_s[1][2] + red_s[1][3]);       // the same in every thread
    if (Z == 0.f) {                   // no part saw a token
        for (int c = c_first; c < nvec; c += c_step) o4[c] = make_float4(0.f, 0.f, 0.f, 0.f);
        if (c_first == 0) lse[r] = -INFINITY;
        return;
    }
    const float L = m + logf(Z);
    for (int j0 = 0; j0 < num_parts; j0 += kMergeThreads) {              // as many parts at a time as there are weights in shared memory
        const int n = min(kMergeThreads, num_parts - j0);
        if (j0 > 0) __syncthreads();
        if (tid < n) w_s[tid] = expf((j0 == 0 ? first : part_lse[(int64_t)(j0 + tid) * rows + r]) - L);
        __syncthreads();
        for (int c = c_first; c < nvec; c += c_step) {
            float4 acc = j0 == 0 ? make_float4(0.f, 0.f, 0.f, 0.f) : o4[c];
            for (int j = 0; j < n; j += kDepth) {
                float4 v[kDepth];
#pragma unroll
                for (int u = 0; u < kDepth; ++u)
                    if (j + u < n) v[u] = reinterpret_cast<const float4 *>(part_out + ((int64_t)(j0 + j + u) * rows + r) * d_v)[c];
#pragma unroll
                for (int u = 0; u < kDepth; ++u) {
                    const float w = j + u < n ? w_s[j + u] : 0.f;
                    if (w != 0.f) {        // (the row of a part without tokens is not looked at)
                        acc.x = fmaf(w, v[u].x, acc.x); acc.y = fmaf(w, v[u].y, acc.y);
                        acc.z = fmaf(w, v[u].z, acc.z); acc.w = fmaf(w, v[u].w, acc.w);
                    }
                }
            }
            o4[c] = acc;
        }
    }
    if (c_first == 0) lse[r] = L;
}

// The combine kernels: block = (entry of the plan's list of split requests, head k of the slice).  A request computed in one
// piece and an empty one were written by the decode kernel itself; a split request is merged from the slots of its workers in
// worker order.  What bounds them is round trips to L2 and DRAM: the list's length and the entry's record come in the first, and the
// record says where the pieces lie, so that their LSEs and their rows come in the second.
constexpr int kMaxParts = 512;     // >= number of workers of any launch (one per SM at most)

// Where a cut request's pieces lie.  Their numbers do not depend on who has made the plan, nor do the sums then: with less cost than workers
// (kGaps: the plan kernel's plans, which may be such), cost unit u is a tile or overhead, and the last worker whose share starts
// at it is number floor(((u + 1) W - 1) / cost).
template <bool kGaps>
struct Pieces {
    int request, first, n, flags, cost, workers;
    __device__ __forceinline__ Pieces(const DecodeParams &p, const int4 &rec)
        : request(rec.x), first(rec.y), n(rec.z - rec.y + 1), flags(rec.w), cost(rec.w >> kSplitCostShift), workers(p.num_workers) {
        if (kGaps && cost > 0) { first = rec.y * cost / workers; n = rec.z * cost / workers - first + 1; }
    }
    __device__ __forceinline__ uint32_t row(int j, int h, int k) const {
        int w = first + j;
        if (kGaps && cost > 0) w = ((w + 1) * workers - 1) / cost;
        return (uint32_t)(2 * w + (j == 0 ? flags & kSplitSecondSlot : 0)) * h + k;
    }
};

// Four columns of a slot's row as they lie in memory.  (Loads first, conversions with the arithmetic: a conversion next to its load would
// make every load wait for the one before it.)
template <bool kF16>
struct PartRow {
    using Raw = typename std::conditional<kF16, uint2, float4>::type;
    static __device__ __forceinline__ Raw load(const DecodeParams &p, uint32_t row, int c) {      // (at most 2 W h rows, of 128 fours)
        return reinterpret_cast<const Raw *>(p.partial_out)[row * (kDV / 4) + c];
    }
    static __device__ __forceinline__ void add(float4 &acc, const Raw &raw, float w) {
        float4 v;
        if constexpr (kF16) {
            const float2 a = __half22float2(*reinterpret_cast<const __half2 *>(&raw.x)), b = __half22float2(*reinterpret_cast<const __half2 *>(&raw.y));
            v = make_float4(a.x, a.y, b.x, b.y);
        } else {
            v = raw;
        }
        acc.x = fmaf(w, v.x, acc.x); acc.y = fmaf(w, v.y, acc.y);
        acc.z = fmaf(w, v.z, acc.z); acc.w = fmaf(w, v.w, acc.w);
    }
};

// kF16: the partial outputs are f16 (rows of 512 halves) or fp32.  kLean: a variant for launches whose requests are cut
// into few pieces each (many requests per worker): at most four part loads in flight, few enough registers for sixteen
// resident blocks per SM instead of eight -- its blocks are short chains of round trips, and what bounds
// the kernel is how many of them an SM holds at a time.
template <bool kF16, bool kLean, bool kGaps>
__global__ void __launch_bounds__(kMergeThreads, kLean ? 16 : 8)
split_combine_kernel(const DecodeParams p, const int4 *split_rec) {
    using Row = PartRow<kF16>;
    __shared__ float w_s[kMaxParts];
    __shared__ uint32_t row_s[kMaxParts];
    __shared__ float sc_s[kF16 ? kMaxParts : 1];      // f16 pieces: the power of two each row was divided by
    __shared__ float red_s[kMergeThreads / 32], sum_s[kMergeThreads / 32];
    const int h = p.head_end - p.head_begin;
    const int k = blockIdx.x % h, entry = blockIdx.x / h;
    const int g = p.head_begin + k;
    grid_launch_dependents();     // a next call's first kernel may come in once every block of this grid has started
    grid_dependency_wait();       // the decode kernel's partial slots (and the plan) are read from here on
    const int n_entries = p.status[8];
    const Pieces<kGaps> pieces(p, split_rec[entry]);          // (unused past the list's end)
    if (entry >= n_entries) return;
    const int i = pieces.request, nparts = pieces.n;
    float4 *o4 = reinterpret_cast<float4 *>(p.out + (int64_t)i * p.out_stride_request + (int64_t)g * p.out_stride_head);
    float *lse = p.lse + (int64_t)i * p.lse_stride_request + g;
    const int c = threadIdx.x;             // 128 threads x float4 = 512 columns
    if (kLean && nparts <= 4) {
        // few pieces, as nearly all requests of such a launch: every thread has all their LSEs, and nothing is exchanged
        typename Row::Raw raw[4];
        float L[4], scale[4];
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            L[j] = -INFINITY; scale[j] = 1.f;
            if (j < nparts) {
                const uint32_t row = pieces.row(j, h, k);
                L[j] = p.partial_lse[row];
                if constexpr (kF16) scale[j] = p.partial_scale[row];
                raw[j] = Row::load(p, row, c);
            }
        }
        const float m = reference_max(fmaxf(fmaxf(L[0], L[1]), fmaxf(L[2], L[3])));
        float Z = 0.f;
#pragma unroll
        for (int j = 0; j < 4; ++j) { L[j] = expf(L[j] - m); Z += L[j]; }      // (0 for a piece that is not there)
        float4 acc = make_float4(0.f, 0.f, 0.f, 0.f);
        if (Z != 0.f) {
            const float inv_z = 1.f / Z;
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                const float w = L[j] * inv_z;
                if (w != 0.f) Row::add(acc, raw[j], kF16 ? w * scale[j] : w);
            }
        }
        o4[c] = acc;
        if (c == 0) *lse = Z == 0.f ? -INFINITY : m + logf(Z);
        return;
    }
    // the first pieces' rows, beside the LSEs
    constexpr int kFirst = kLean ? 0 : kF16 ? 16 : 8;
    typename Row::Raw first[kFirst + 1];
#pragma unroll
    for (int u = 0; u < kFirst; ++u)
        if (u < nparts) first[u] = Row::load(p, pieces.row(u, h, k), c);
    float m = -INFINITY;
    for (int j = c; j < nparts; j += kMergeThreads) {
        const uint32_t row = pieces.row(j, h, k);
        const float L = p.partial_lse[row];
        if constexpr (kF16) sc_s[j] = p.partial_scale[row];
        w_s[j] = L; row_s[j] = row;
        m = fmaxf(m, L);
    }
    for (int o = 16; o; o >>= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, o));
    if ((c & 31) == 0) red_s[c >> 5] = m;
    __syncthreads();
    m = reference_max(fmaxf(fmaxf(red_s[0], red_s[1]), fmaxf(red_s[2], red_s[3])));
    float Z = 0.f;
    for (int j = c; j < nparts; j += kMergeThreads) { w_s[j] = expf(w_s[j] - m); Z += w_s[j]; }     // (0 for a piece that saw no token)
    for (int o = 16; o; o >>= 1) Z += __shfl_xor_sync(0xffffffffu, Z, o);
    if ((c & 31) == 0) sum_s[c >> 5] = Z;
    __syncthreads();
    Z = (sum_s[0] + sum_s[1]) + (sum_s[2] + sum_s[3]);     // the same in every thread
    if (Z == 0.f) {                        // no piece saw a token (a query row whose causal range is empty)
        o4[c] = make_float4(0.f, 0.f, 0.f, 0.f);
        if (c == 0) *lse = -INFINITY;
        return;
    }
    const float inv_z = 1.f / Z;
    float4 acc = make_float4(0.f, 0.f, 0.f, 0.f);
    auto add = [&](int j, const typename Row::Raw &raw) {
        float w = w_s[j] * inv_z;
        if (w != 0.f) {                    // (0: a piece that saw no token)
            if constexpr (kF16) w *= sc_s[j];
            Row::add(acc, raw, w);
        }
    };
#pragma unroll
    for (int u = 0; u < kFirst; ++u)
        if (u < nparts) add(u, first[u]);
    int j = kFirst;
    // sixteen, then (up to) four part loads in flight per thread: one long context cut into a piece per worker is merged by
    // one block per head, and the part loop is a chain of round trips to L2 / HBM
    for (; !kLean && j + 16 <= nparts; j += 16) {
        typename Row::Raw raw[16];
#pragma unroll
        for (int u = 0; u < 16; ++u) raw[u] = Row::load(p, row_s[j + u], c);
#pragma unroll
        for (int u = 0; u < 16; ++u) add(j + u, raw[u]);
    }
    // (loads first: a request cut into two or three pieces, the usual case, would pay a round trip per piece)
    for (; j < nparts; j += 4) {
        typename Row::Raw raw[4];
#pragma unroll
        for (int u = 0; u < 4; ++u)
            if (j + u < nparts) raw[u] = Row::load(p, row_s[j + u], c);
#pragma unroll
        for (int u = 0; u < 4; ++u)
            if (j + u < nparts) add(j + u, raw[u]);
    }
    o4[c] = acc;
    if (c == 0) *lse = m + logf(Z);
}

// The same for launches of no more rows than SMs (a small batch): four groups of 128 threads take every fourth piece and add
// their sums in shared memory.  Behind the kernels of 16 and 32 heads 2 KB of shared memory and 32 registers, so that a block fits
// beside a decode CTA of 16 heads: the next call's CTAs come in, plan and prefetch while this kernel runs (eight layers of 8 requests:
// with the kernel above, 6 KB a block, they came in 1.6 to 4.4 us later, one by one as its blocks left; with 40 registers too); the pieces' rows wait
// in shared memory then (worked out where they are loaded, they did not fit those registers: one context of 16,384 tokens on 16 heads 18.4 us,
// now 17.1; of 65,536 28.9 and 27.5).  Behind the
// others (kDeep), which leave no room for that anyway, more loads are in flight, the first of them beside those of the LSEs: 74
// pieces on 128 heads 5.4 us, now 4.5.  (A warp for itself with 32 columns of a row and no barriers: 10 us, every warp loads all LSEs then.)
constexpr int kGroupedParts = 160, kCombineGroups = 4;
template <bool kF16, bool kDeep, bool kGaps>
__global__ void __launch_bounds__(kCombineGroups * kMergeThreads, kDeep ? 2 : 4)
grouped_combine_kernel(const DecodeParams p, const int4 *split_rec) {
    using Row = PartRow<kF16>;
    constexpr int kThreads = kCombineGroups * kMergeThreads, kDepth = !kDeep ? 4 : kF16 ? 16 : 8;
    // weights (f16 pieces: times the power of two each row was divided by) and (!kDeep) row numbers; then the groups' sums
    __shared__ __align__(16) float smem_f[4 * kMergeThreads];
    static_assert(2 * kGroupedParts <= 4 * kMergeThreads && kGroupedParts <= kThreads, "a piece per thread");
    __shared__ float max_s[kThreads / 32], sum_s[kThreads / 32];
    float *const w_s = smem_f;
    uint32_t *const row_s = reinterpret_cast<uint32_t *>(smem_f + kGroupedParts);
    const int h = p.head_end - p.head_begin;
    const int k = blockIdx.x % h, entry = blockIdx.x / h;
    const int g = p.head_begin + k;
    grid_launch_dependents();
    grid_dependency_wait();
    const int n_entries = p.status[8];
    const Pieces<kGaps> pieces(p, split_rec[entry]);
    if (entry >= n_entries) return;
    const int i = pieces.request, nparts = pieces.n;
    float4 *o4 = reinterpret_cast<float4 *>(p.out + (int64_t)i * p.out_stride_request + (int64_t)g * p.out_stride_head);
    float *lse = p.lse + (int64_t)i * p.lse_stride_request + g;
    const int tid = threadIdx.x, c = tid % kMergeThreads, group = tid / kMergeThreads;
    float L = -INFINITY, scale = 1.f;
    if (tid < nparts) {
        const uint32_t row = pieces.row(tid, h, k);
        L = p.partial_lse[row];
        if constexpr (kF16) scale = p.partial_scale[row];
        if constexpr (!kDeep) row_s[tid] = row;
    }
    typename Row::Raw raw[kDepth];
    auto load = [&](int j0) {
#pragma unroll
        for (int u = 0; u < kDepth; ++u) {
            const int j = j0 + u * kCombineGroups;
            if (j < nparts) raw[u] = Row::load(p, kDeep ? pieces.row(j, h, k) : row_s[j], c);
        }
    };
    if constexpr (kDeep) load(group);
    float m = L;
    for (int o = 16; o; o >>= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, o));
    if ((tid & 31) == 0) max_s[tid >> 5] = m;
    __syncthreads();
    m = max_s[0];
#pragma unroll
    for (int x = 1; x < kThreads / 32; ++x) m = fmaxf(m, max_s[x]);
    m = reference_max(m);
    float Z = tid < nparts ? expf(L - m) : 0.f;
    if (tid < nparts) w_s[tid] = Z * scale;
    for (int o = 16; o; o >>= 1) Z += __shfl_xor_sync(0xffffffffu, Z, o);
    if ((tid & 31) == 0) sum_s[tid >> 5] = Z;
    __syncthreads();
    Z = sum_s[0];
#pragma unroll
    for (int x = 1; x < kThreads / 32; ++x) Z += sum_s[x];       // same order in every thread: one value of Z
    if (Z == 0.f) {                        // no piece saw a token
        if (group == 0) o4[c] = make_float4(0.f, 0.f, 0.f, 0.f);
        if (tid == 0) *lse = -INFINITY;
        return;
    }
    const float inv_z = 1.f / Z;
    float4 acc = make_float4(0.f, 0.f, 0.f, 0.f);
    for (int j0 = group; j0 < nparts; j0 += kCombineGroups * kDepth) {
        if (!kDeep || j0 != group) load(j0);
#pragma unroll
        for (int u = 0; u < kDepth; ++u) {
            const int j = j0 + u * kCombineGroups;
            const float w = j < nparts ? w_s[j] * inv_z : 0.f;
            if (w != 0.f) Row::add(acc, raw[u], w);              // (0: a piece that saw no token)
        }
    }
    float4 *const total = reinterpret_cast<float4 *>(smem_f);
    __syncthreads();                       // the weights have been read
#pragma unroll 1
    for (int x = kCombineGroups - 1; x >= 0; --x) {
        if (group == x) {
            if (x < kCombineGroups - 1) {
                const float4 v = total[c];
                acc.x += v.x; acc.y += v.y; acc.z += v.z; acc.w += v.w;
            }
            if (x > 0) total[c] = acc;
            else o4[c] = acc;
        }
        if (x > 0) __syncthreads();
    }
    if (tid == 0) *lse = m + logf(Z);
}

}  // namespace

cudaError_t launch_lse_merge(int num_parts, int64_t rows, int d_v, const float *part_out,
                             const float *part_lse, float *out, float *lse, int sm_count, cudaStream_t stream) {
    const int64_t wide = (d_v / 4 + kMergeThreads - 1) / kMergeThreads;
    const int64_t resident = 8 * (int64_t)sm_count;       // (24,960 rows of five parts, a decode in front: 121.6 us with eight loads, now 111)
    // Rows are cut while there are too few of them to fill the SMs, into about two blocks for each place.  More rows than places gain
    // nothing from it and each block starts with the row's weights: 3,000 rows of two parts, 1,536 wide, 7.9 us whole and 12.1 cut.
    const int64_t cut = rows > 0 && rows <= resident ? (2 * resident + rows - 1) / rows : 1;
    const dim3 grid((unsigned)rows, (unsigned)(cut < wide ? cut : wide));
    const cudaError_t e = launch_dependent(rows * grid.y <= resident ? lse_merge_kernel<8> : lse_merge_kernel<4>, grid, dim3(kMergeThreads), 0, stream, num_parts, rows, d_v,
                                           part_out, part_lse, out, lse);
    count_launch();
    return e;
}

cudaError_t launch_split_combine(const DecodeParams &p, const int4 *split_rec, int sm_count, cudaStream_t stream) {
    // at most one request straddles each boundary between consecutive workers
    const int max_split = p.num_workers < p.B ? p.num_workers : p.B;
    dim3 grid((unsigned)((int64_t)(p.head_end - p.head_begin) * max_split));
    // many requests per worker: every request is cut into a few pieces at most
    const bool lean = (int64_t)p.B * 4 >= p.num_workers;
    const bool room = p.heads_per_group <= 32 && p.num_groups == 1;       // for a block beside a decode CTA
    // as many rows as are resident at once (room: one beside each CTA): two requests on 128 heads 17.8 us, now 16.1; with 384 rows 18.0 against 17.4
    const bool grouped = !lean && grid.x <= (room ? 1u : 2u) * (unsigned)sm_count && p.num_workers <= kGroupedParts;
    auto choose = [&](auto gaps) {
        constexpr bool kGaps = decltype(gaps)::value;
        return grouped ? (p.partial_f16 ? grouped_combine_kernel<true, true, kGaps> : room ? grouped_combine_kernel<false, false, kGaps> : grouped_combine_kernel<false, true, kGaps>)
             : p.partial_f16 ? (lean ? split_combine_kernel<true, true, kGaps> : split_combine_kernel<true, false, kGaps>)
                             : (lean ? split_combine_kernel<false, true, kGaps> : split_combine_kernel<false, false, kGaps>);
    };
    const bool gaps = p.plan_mode == kPlanWorkspace;
    auto kernel = gaps ? choose(std::true_type()) : choose(std::false_type());
    // the decode kernel's shared-memory carve-out is kept (a preference: a failure is not an error)
    static DeviceOnce once[2][2][2][2];
    once[gaps][grouped][p.partial_f16 != 0][grouped ? room : lean].run([&] {
        cudaFuncSetAttribute(kernel, cudaFuncAttributePreferredSharedMemoryCarveout, cudaSharedmemCarveoutMaxShared);
        return cudaSuccess;
    });
    cudaError_t e = launch_dependent(kernel, grid, dim3(grouped ? kCombineGroups * kMergeThreads : kMergeThreads), 0, stream, p, split_rec);
    count_launch();
    return e;
}

}  // namespace splash
