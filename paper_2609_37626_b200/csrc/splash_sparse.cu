// Sparse decode on the fp32 kernel (SPLASH_FLAG_SIMT): the listed rows of every request gathered into a dense, request-major
// bf16 cache in the workspace, over which that kernel then runs with the list lengths as context lengths.  (The tensor-core
// kernels gather their rows themselves, splash_gather.cuh.)  A warp takes four rows at a time.
#include "splash_gather.cuh"

namespace splash {

namespace {

constexpr int kGatherThreads = 256;

__global__ void __launch_bounds__(kGatherThreads)
sparse_gather_kernel(int B, int max_sel, int pages_per_request, const uint8_t *__restrict__ kv_pool, int num_pool_pages,
                     const int32_t *__restrict__ block_table, int64_t table_stride, const int32_t *__restrict__ seq_lens,
                     const int32_t *__restrict__ sel, int64_t sel_stride, const int32_t *__restrict__ sel_count,
                     uint8_t *__restrict__ dense_pool, int32_t *__restrict__ dense_table) {
    const int64_t thread = (int64_t)blockIdx.x * kGatherThreads + threadIdx.x, threads = (int64_t)gridDim.x * kGatherThreads;
    const int slots_per_request = pages_per_request * kPage, x = threadIdx.x & 7;
    // the dense cache's page table (its context lengths are the list counts, read by the plan)
    for (int64_t e = thread; e < (int64_t)B * pages_per_request; e += threads) dense_table[e] = (int32_t)e;
    // eight lanes a row: 16 codes of each of its four blocks, 16 bytes of its rope part
    for (int64_t slot = thread >> 3; slot < (int64_t)B * slots_per_request; slot += threads >> 3) {
        const int req = (int)(slot / slots_per_request), idx = (int)(slot % slots_per_request);
        const int cnt = sel_count[req];
        const bool bad_count = cnt < 0 || cnt > max_sel;       // stands for one poisoned row, as in the plan
        unsigned long long row = gather::kSkip;
        if (idx < (bad_count ? 1 : cnt)) {
            const int tok = bad_count ? -1 : sel[(int64_t)req * sel_stride + idx];
            const int page = tok >= 0 && tok < seq_lens[req] ? block_table[(int64_t)req * table_stride + tok / kPage] : -1;
            row = page < 0 || page >= num_pool_pages ? gather::kPoison
                : reinterpret_cast<unsigned long long>(kv_pool + ((int64_t)page * kPage + tok % kPage) * kSparseRowBytes);
        }
        uint8_t *const dst = dense_pool + slot * (kDQK * 2);
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            const uint4 c = gather::load16(row, 128 * j + 16 * x, gather::kPoisonCodes);
            const float s = row > gather::kPoison ? reinterpret_cast<const float *>(row + kDLatent)[j] : 1.f;
            gather::dequant16(c, s, dst + (128 * j + 16 * x) * 2, 0, 0);
        }
        *reinterpret_cast<uint4 *>(dst + kDLatent * 2 + 16 * x) = gather::load16(row, kDLatent + 16 + 16 * x, gather::kPoisonRope);
    }
}

}  // namespace

cudaError_t launch_sparse_gather(int B, int max_sel, int pages_per_request, const void *kv_pool, int num_pool_pages,
                                 const int32_t *block_table, int64_t table_stride, const int32_t *seq_lens,
                                 const int32_t *sel, int64_t sel_stride, const int32_t *sel_count, void *dense_pool,
                                 int32_t *dense_table, int sm_count, cudaStream_t stream) {
    const int64_t rows = (int64_t)B * pages_per_request * kPage, per_block = kGatherThreads / 8;
    int64_t blocks = (rows + per_block - 1) / per_block;
    const int64_t cap = (int64_t)sm_count * 8;          // resident blocks; the loop strides over the rest
    if (blocks > cap) blocks = cap;
    if (blocks < 1) blocks = 1;
    sparse_gather_kernel<<<(unsigned)blocks, kGatherThreads, 0, stream>>>(
        B, max_sel, pages_per_request, static_cast<const uint8_t *>(kv_pool), num_pool_pages, block_table, table_stride, seq_lens, sel,
        sel_stride, sel_count, static_cast<uint8_t *>(dense_pool), dense_table);
    count_launch();
    return cudaGetLastError();
}

}  // namespace splash
