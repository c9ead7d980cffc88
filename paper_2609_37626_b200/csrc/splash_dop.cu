// DOP transfer layout changes (App. E): the regrouping kernels on either side of the two
// all-to-alls that turn a tensor in global-row, local-head order into owner-row, all-head
// order and back.  Whole rows of bytes are moved, nothing is computed: byte-exact.
//
//   pack_rows     send[p][j][0 .. da + db) = a[send_row[p]][j][0 .. da) ++ b[send_row[p]][j][0 .. db)
//                 (rows grouped by destination owner; the no-position and the rotary part of the query
//                 are fused into one row so that one collective moves both)
//   unpack_rows   out[send_row[p]][j][:] = recv[p][j][:]                  (the reverse exchange's last step)
//   swap_outer    out[r][s][:] = in[s][r][:]        ([T][n][h][d] <-> [n][T][h][d]: source-rank-major receive
//                 buffer to all-head order, head s * h + j from rank s, and its inverse)
//
// Each has a 32- and a 16-byte vector path (all base pointers, row pitches and part lengths multiples of it) and a 2-byte
// scalar fallback.  HBM-bound: bytes read + bytes written.
#include <type_traits>

#include "splash_copy.cuh"

namespace splash {

namespace {

// A position: h rows of va + vb vectors.
template <typename Vec, bool kBlock>
__global__ void __launch_bounds__(kCopyThreads, 4)
pack_rows_kernel(const Vec *a, const Vec *b, Vec *out, const int32_t *send_row, int64_t n,
                 const RowSplit split, int va, int vb, int64_t a_row_pitch, int64_t a_head_pitch, int64_t b_row_pitch, int64_t b_head_pitch) {
    grid_dependency_wait();       // launched while the work before it on the stream still runs
    grid_launch_dependents();
    const unsigned vrow = (unsigned)(va + vb);     // vectors per (position, head); below 2^31
    own_row<kBlock>(split, n, [&](int64_t p, int64_t first, int vecs) {
        const int64_t src = send_row[p], j0 = kBlock && first > 0 ? first / vrow : 0;
        const unsigned at = (unsigned)(first - j0 * vrow);
        const Vec *const pa = a + src * a_row_pitch + j0 * a_head_pitch, *const pb = b + src * b_row_pitch + j0 * b_head_pitch;
        copy_row<kBlock>(out + p * split.vecs + first, vecs, split.group, [&](int i) {
            const unsigned t = at + (unsigned)i;
            const int j = (int)(t / vrow), c = (int)(t - (unsigned)j * vrow);
            return c < va ? pa + j * a_head_pitch + c : pb + j * b_head_pitch + (c - va);
        });
    });
}

template <typename Vec, bool kBlock>
__global__ void __launch_bounds__(kCopyThreads, 4)
unpack_rows_kernel(const Vec *recv, Vec *out, const int32_t *send_row, int64_t n, const RowSplit split,
                   int64_t out_row_pitch) {
    grid_dependency_wait();
    grid_launch_dependents();
    own_row<kBlock>(split, n, [&](int64_t p, int64_t first, int vecs) {
        const Vec *const src = recv + p * split.vecs + first;
        copy_row<kBlock>(out + send_row[p] * out_row_pitch + first, vecs, split.group, [&](int c) { return src + c; });
    });
}

// block (s, r) of `split.vecs` vectors moves from in[s][r] to out[r][s]
template <typename Vec, bool kBlock>
__global__ void __launch_bounds__(kCopyThreads, 4)
swap_outer_kernel(const Vec *in, Vec *out, int64_t A, int64_t Bn, const RowSplit split) {
    grid_dependency_wait();
    grid_launch_dependents();
    own_row<kBlock>(split, A * Bn, [&](int64_t blk, int64_t first, int vecs) {
        const int64_t s = (uint64_t)(blk | Bn) >> 32 ? blk / Bn : (int64_t)((uint32_t)blk / (uint32_t)Bn), r = blk - s * Bn;
        const Vec *const src = in + blk * split.vecs + first;
        copy_row<kBlock>(out + (r * A + s) * split.vecs + first, vecs, split.group, [&](int c) { return src + c; });
    });
}

}  // namespace

// `launch` for the vector type of the width and for blocks or groups
template <typename Launch>
static cudaError_t launch_rows(int width, int64_t rows, int64_t row_bytes, int sm_count, Launch &&launch) {
    const RowSplit split(rows, row_bytes / width, width, sm_count);
    if (split.items > 0x7fffffff) return cudaErrorInvalidValue;      // (rows of 200 GB and more)
    auto with = [&](auto vec) {
        return split.group == kCopyThreads ? launch(vec, split, std::true_type{}) : launch(vec, split, std::false_type{});
    };
    const cudaError_t e = width == 32 ? with(Vec32{}) : width == 16 ? with(uint4{}) : with(uint16_t{});
    count_launch();
    return e;
}

cudaError_t launch_dop_pack_rows(const void *a, const void *b, void *out, const int32_t *send_row, int64_t n, int h,
                                 int64_t a_bytes, int64_t b_bytes, int64_t a_row_pitch, int64_t a_head_pitch,
                                 int64_t b_row_pitch, int64_t b_head_pitch, int sm_count, cudaStream_t stream) {
    const int width = copy_width(address_bits(a) | address_bits(b) | address_bits(out) | (uint64_t)(a_bytes | b_bytes | a_row_pitch | a_head_pitch |
                                                                                                   b_row_pitch | b_head_pitch));
    if ((a_bytes + b_bytes) / width > 0x7fffffff) return cudaErrorInvalidValue;      // more vectors per head than an int counts
    return launch_rows(width, n, h * (a_bytes + b_bytes), sm_count, [&](auto vec, const RowSplit &split, auto block) {
        using Vec = decltype(vec);
        constexpr int64_t kW = sizeof(Vec);
        return launch_dependent(pack_rows_kernel<Vec, decltype(block)::value>, dim3((unsigned)split.items), dim3(kCopyThreads), 0, stream,
                                static_cast<const Vec *>(a), static_cast<const Vec *>(b), static_cast<Vec *>(out), send_row, n, split,
                                (int)(a_bytes / kW), (int)(b_bytes / kW), a_row_pitch / kW, a_head_pitch / kW, b_row_pitch / kW, b_head_pitch / kW);
    });
}

cudaError_t launch_dop_unpack_rows(const void *recv, void *out, const int32_t *send_row, int64_t n, int64_t row_bytes,
                                   int64_t out_row_pitch, int sm_count, cudaStream_t stream) {
    const int width = copy_width(address_bits(recv) | address_bits(out) | (uint64_t)(row_bytes | out_row_pitch));
    return launch_rows(width, n, row_bytes, sm_count, [&](auto vec, const RowSplit &split, auto block) {
        using Vec = decltype(vec);
        return launch_dependent(unpack_rows_kernel<Vec, decltype(block)::value>, dim3((unsigned)split.items), dim3(kCopyThreads), 0, stream,
                                static_cast<const Vec *>(recv), static_cast<Vec *>(out), send_row, n, split, out_row_pitch / (int64_t)sizeof(Vec));
    });
}

cudaError_t launch_dop_swap_outer(const void *in, void *out, int64_t A, int64_t Bn, int64_t inner_bytes, int sm_count, cudaStream_t stream) {
    const int width = copy_width(address_bits(in) | address_bits(out) | (uint64_t)inner_bytes);
    return launch_rows(width, A * Bn, inner_bytes, sm_count, [&](auto vec, const RowSplit &split, auto block) {
        using Vec = decltype(vec);
        return launch_dependent(swap_outer_kernel<Vec, decltype(block)::value>, dim3((unsigned)split.items), dim3(kCopyThreads), 0, stream,
                                static_cast<const Vec *>(in), static_cast<Vec *>(out), A, Bn, split);
    });
}

}  // namespace splash
