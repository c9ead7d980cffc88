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
#include "splash_copy.cuh"

namespace splash {

namespace {

// One position per block: h rows of va + vb vectors.
template <typename Vec>
__global__ void __launch_bounds__(kCopyThreads, 4)
pack_rows_kernel(const Vec *__restrict__ a, const Vec *__restrict__ b, Vec *__restrict__ out, const int32_t *__restrict__ send_row,
                 int h, int va, int vb, int64_t a_row_pitch, int64_t a_head_pitch, int64_t b_row_pitch, int64_t b_head_pitch) {
    grid_dependency_wait();       // launched while the work before it on the stream still runs
    grid_launch_dependents();
    const int64_t p = blockIdx.x, src = send_row[p];
    const unsigned vrow = (unsigned)(va + vb);     // vectors per (position, head)
    a += src * a_row_pitch;
    b += src * b_row_pitch;
    copy_row(out + p * h * (int64_t)vrow, h * (int)vrow, [&](int i) {
        const int j = (int)((unsigned)i / vrow), c = i - j * (int)vrow;
        return c < va ? a + j * a_head_pitch + c : b + j * b_head_pitch + (c - va);
    });
}

template <typename Vec>
__global__ void __launch_bounds__(kCopyThreads, 4)
unpack_rows_kernel(const Vec *__restrict__ recv, Vec *__restrict__ out, const int32_t *__restrict__ send_row, int64_t n, int64_t per_pos,
                   int64_t out_row_pitch) {
    grid_dependency_wait();
    grid_launch_dependents();
    for (int64_t p = blockIdx.x; p < n; p += gridDim.x) {
        const int64_t dst = send_row[p];
        // (a row of more vectors than an int counts goes in pieces)
        for (int64_t c0 = 0; c0 < per_pos; c0 += 1 << 30) {
            const Vec *src = recv + p * per_pos + c0;
            copy_row(out + dst * out_row_pitch + c0, (int)(per_pos - c0 < (1 << 30) ? per_pos - c0 : 1 << 30), [&](int c) { return src + c; });
        }
    }
}

// block (s, r) of `inner` vectors moves from in[s][r] to out[r][s]
template <typename Vec>
__global__ void __launch_bounds__(kCopyThreads, 4)
swap_outer_kernel(const Vec *__restrict__ in, Vec *__restrict__ out, int64_t A, int64_t Bn, int64_t inner) {
    grid_dependency_wait();
    grid_launch_dependents();
    for (int64_t blk = blockIdx.x; blk < A * Bn; blk += gridDim.x) {
        const int64_t s = blk / Bn, r = blk - s * Bn;
        for (int64_t c0 = 0; c0 < inner; c0 += 1 << 30) {
            const Vec *src = in + blk * inner + c0;
            copy_row(out + (r * A + s) * inner + c0, (int)(inner - c0 < (1 << 30) ? inner - c0 : 1 << 30), [&](int c) { return src + c; });
        }
    }
}

}  // namespace

cudaError_t launch_dop_pack_rows(const void *a, const void *b, void *out, const int32_t *send_row, int64_t n, int h,
                                 int64_t a_bytes, int64_t b_bytes, int64_t a_row_pitch, int64_t a_head_pitch,
                                 int64_t b_row_pitch, int64_t b_head_pitch, cudaStream_t stream) {
    auto launch = [&](auto vec) {
        using Vec = decltype(vec);
        constexpr int64_t kW = sizeof(Vec);
        return launch_dependent(pack_rows_kernel<Vec>, dim3((unsigned)n), dim3(kCopyThreads), 0, stream, static_cast<const Vec *>(a),
                                static_cast<const Vec *>(b), static_cast<Vec *>(out), send_row, h, (int)(a_bytes / kW), (int)(b_bytes / kW),
                                a_row_pitch / kW, a_head_pitch / kW, b_row_pitch / kW, b_head_pitch / kW);
    };
    const int width = copy_width(address_bits(a) | address_bits(b) | address_bits(out) | (uint64_t)(a_bytes | b_bytes | a_row_pitch | a_head_pitch |
                                                                                                   b_row_pitch | b_head_pitch));
    const cudaError_t e = width == 32 ? launch(Vec32{}) : width == 16 ? launch(uint4{}) : launch(uint16_t{});
    count_launch();
    return e;
}

cudaError_t launch_dop_unpack_rows(const void *recv, void *out, const int32_t *send_row, int64_t n, int64_t row_bytes,
                                   int64_t out_row_pitch, cudaStream_t stream) {
    auto launch = [&](auto vec) {
        using Vec = decltype(vec);
        constexpr int64_t kW = sizeof(Vec);
        return launch_dependent(unpack_rows_kernel<Vec>, dim3((unsigned)(n < 0x7fffffffLL ? n : 0x7fffffffLL)), dim3(kCopyThreads), 0, stream,
                                static_cast<const Vec *>(recv), static_cast<Vec *>(out), send_row, n, row_bytes / kW, out_row_pitch / kW);
    };
    const int width = copy_width(address_bits(recv) | address_bits(out) | (uint64_t)(row_bytes | out_row_pitch));
    const cudaError_t e = width == 32 ? launch(Vec32{}) : width == 16 ? launch(uint4{}) : launch(uint16_t{});
    count_launch();
    return e;
}

cudaError_t launch_dop_swap_outer(const void *in, void *out, int64_t A, int64_t Bn, int64_t inner_bytes, cudaStream_t stream) {
    const int64_t blocks = A * Bn;
    auto launch = [&](auto vec) {
        using Vec = decltype(vec);
        return launch_dependent(swap_outer_kernel<Vec>, dim3((unsigned)(blocks < 0x7fffffffLL ? blocks : 0x7fffffffLL)), dim3(kCopyThreads), 0,
                                stream, static_cast<const Vec *>(in), static_cast<Vec *>(out), A, Bn, inner_bytes / (int64_t)sizeof(Vec));
    };
    const int width = copy_width(address_bits(in) | address_bits(out) | (uint64_t)inner_bytes);
    const cudaError_t e = width == 32 ? launch(Vec32{}) : width == 16 ? launch(uint4{}) : launch(uint16_t{});
    count_launch();
    return e;
}

}  // namespace splash
