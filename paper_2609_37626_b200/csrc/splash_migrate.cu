// KV page migration between two page pools in HBM, with block-table rewrite: the
// single-GPU part of a layout switch (kept blocks are repacked into the destination
// view; the table is the page metadata that must follow them).  Byte-exact.
#include "splash_copy.cuh"

namespace splash {

namespace {

constexpr int kScaleVecs = kPage * 4 / 16;  // 16-byte vectors of a scale page

// Entry s of the remap table: which listed page has the table id s.  The table is not cleared first (that was a kernel of
// its own): an entry nobody wrote in this call holds anything, and the rewrite believes an entry only if the page that it
// names does have that id.
__global__ void __launch_bounds__(kCopyThreads)
remap_scatter_kernel(int32_t *remap, const int32_t *src_ids, int64_t n, int32_t src_base, int32_t max_page_id) {
    grid_dependency_wait();         // launched while the work before it on the stream still runs
    grid_launch_dependents();       // the copy's blocks may come in; they wait for this grid
    const int64_t j = (int64_t)blockIdx.x * kCopyThreads + threadIdx.x;
    if (j < n) {
        const int32_t s = src_base + src_ids[j];
        if (s >= 0 && s < max_page_id) remap[s] = (int32_t)j;
    }
}

struct MigrateParams {
    const void *src_pool;
    void *dst_pool;
    const uint4 *src_scales;
    uint4 *dst_scales;
    int64_t page_bytes;
    const int32_t *src_ids, *dst_ids;
    int32_t n, src_base, dst_base, max_page_id;
    int32_t parts;                   // blocks per page, `per` vectors each
    int64_t vecs, per;
    int32_t *table;
    const int32_t *remap;
    int64_t num_entries;
    int32_t table_blocks, spacing;   // block r * spacing, r < table_blocks, rewrites a piece of the table, the others copy pages
};

constexpr int kEntriesPerBlock = kCopyThreads * 4;

__device__ __forceinline__ void rewrite_entries(const MigrateParams &p, int64_t piece) {
    int64_t e[4];
    int32_t id[4], j[4];
    // four chains of table entry -> page -> its ids per thread, a round trip for each link of all four
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        e[k] = piece * kEntriesPerBlock + k * kCopyThreads + threadIdx.x;
        id[k] = e[k] < p.num_entries ? p.table[e[k]] : -1;
    }
#pragma unroll
    for (int k = 0; k < 4; ++k) j[k] = id[k] >= 0 && id[k] < p.max_page_id ? p.remap[id[k]] : -1;
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        if (j[k] < 0 || j[k] >= p.n) continue;
        const int32_t s = p.src_base + p.src_ids[j[k]], d = p.dst_base + p.dst_ids[j[k]];
        if (s == id[k] && d >= 0) p.table[e[k]] = d;
    }
}

// One block per page, several for a large one (RowSplit), the first with its scale page, and the table's rewrite in blocks spread evenly between them.  Bound by HBM.
template <typename Vec>
__global__ void __launch_bounds__(kCopyThreads, 4)
page_migrate_kernel(const __grid_constant__ MigrateParams p) {
    // Every block, those that copy too: that the scatter kernel has waited for the work in front says nothing to a block that does not.
    grid_dependency_wait();
    grid_launch_dependents();
    const int b = blockIdx.x;
    const int before = min(p.table_blocks, b / p.spacing + 1);     // table blocks up to and including this place
    if (b % p.spacing == 0 && b / p.spacing < p.table_blocks) {
        rewrite_entries(p, b / p.spacing);
        return;
    }
    const int x = b - before, j = p.parts == 1 ? x : x / p.parts;
    const int64_t first = p.parts == 1 ? 0 : (x - j * p.parts) * p.per;
    const int64_t s = p.src_ids[j], d = p.dst_ids[j];
    const Vec *src = reinterpret_cast<const Vec *>(static_cast<const char *>(p.src_pool) + s * p.page_bytes) + first;
    Vec *dst = reinterpret_cast<Vec *>(static_cast<char *>(p.dst_pool) + d * p.page_bytes) + first;
    const int count = p.parts == 1 ? (int)p.vecs : (int)min(p.per, p.vecs - first);      // (none at the end of some)
    copy_row<true>(dst, count, kCopyThreads, [&](int c) { return src + c; });
    if (first > 0) return;
    if (p.src_scales != nullptr && threadIdx.x < kScaleVecs)
        p.dst_scales[d * kScaleVecs + threadIdx.x] = p.src_scales[s * kScaleVecs + threadIdx.x];
}

// Remap table of the allocation-free entry point: lives in the library's device image,
// one copy on every GPU that loads it, until the process exits.
static __device__ __align__(256) int32_t g_static_remap[kStaticMigrateMaxPageId];

}  // namespace

// Device address of g_static_remap on the current device.  In host code the array's
// name only stands for the symbol; the address a kernel can use comes from
// cudaGetSymbolAddress, looked up once per device with that device current.
// The per-device cache is filled under a lock, so that two host threads making their first call on a device at the
// same time do not race on it (both would store the same address, but the lock costs nothing next to a launch).
cudaError_t static_remap_address(int32_t **ptr) {
    static int32_t *cache[64] = {nullptr};
    static std::mutex mu;
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    if (dev < 0 || dev >= 64) return cudaErrorInvalidDevice;
    std::lock_guard<std::mutex> lock(mu);
    if (cache[dev] == nullptr) {
        void *addr = nullptr;
        e = cudaGetSymbolAddress(&addr, g_static_remap);
        if (e != cudaSuccess) return e;
        cache[dev] = static_cast<int32_t *>(addr);
    }
    *ptr = cache[dev];
    return cudaSuccess;
}

cudaError_t launch_page_migrate(const void *src_pool, const float *src_scales, void *dst_pool,
                                float *dst_scales, int64_t page_bytes, const int32_t *src_ids,
                                const int32_t *dst_ids, int64_t n, int32_t src_base, int32_t dst_base,
                                int32_t max_page_id, int32_t *block_table, int64_t num_entries,
                                int32_t *remap, int sm_count, cudaStream_t stream) {
    MigrateParams p;
    p.src_pool = src_pool; p.dst_pool = dst_pool;
    p.src_scales = reinterpret_cast<const uint4 *>(src_scales); p.dst_scales = reinterpret_cast<uint4 *>(dst_scales);
    p.page_bytes = page_bytes; p.src_ids = src_ids; p.dst_ids = dst_ids; p.n = (int32_t)n;
    p.src_base = src_base; p.dst_base = dst_base; p.max_page_id = max_page_id;
    p.table = block_table; p.remap = remap; p.num_entries = num_entries;
    const bool table = num_entries > 0 && max_page_id > 0;
    p.table_blocks = table ? (int32_t)((num_entries + kEntriesPerBlock - 1) / kEntriesPerBlock) : 0;
    // (in 32-byte vectors where the pages lie on 32-byte boundaries: they do in every pool of whole pages whose base does)
    const bool wide = copy_width(address_bits(src_pool) | address_bits(dst_pool) | (uint64_t)page_bytes) == 32;
    const RowSplit split(n, page_bytes / (wide ? 32 : 16), wide ? 32 : 16, sm_count);
    p.parts = split.parts; p.vecs = split.vecs; p.per = split.per;
    const int64_t blocks = n * p.parts + p.table_blocks;
    p.spacing = p.table_blocks > 0 ? (int32_t)(blocks / p.table_blocks) : 1;
    cudaError_t e = cudaSuccess;
    if (table) {
        e = launch_dependent(remap_scatter_kernel, dim3((unsigned)((n + kCopyThreads - 1) / kCopyThreads)), dim3(kCopyThreads), 0, stream,
                             remap, src_ids, n, src_base, max_page_id);
        count_launch();
        if (e != cudaSuccess) return e;
    }
    e = launch_dependent(wide ? page_migrate_kernel<Vec32> : page_migrate_kernel<uint4>, dim3((unsigned)blocks), dim3(kCopyThreads), 0, stream, p);
    count_launch();
    return e;
}

}  // namespace splash
