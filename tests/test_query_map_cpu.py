"""The tensor map of the query rows is a way of loading them, not a condition of the call: where there is none, whether the strides rule
it out or the encoder does, the rows come by other loads and no error is left behind.  The launcher's own host code, with an encoder
that notes what it is asked."""
import os
import subprocess

from paper_2609_37626_b200 import build

PROGRAM = r"""
#include <cuda.h>
#include <cuda_runtime.h>
#include <cstdio>
#include <cstring>
static int asked, errors;
static CUresult answer;
static cuuint64_t strides[3];
static CUresult encode(CUtensorMap *, CUtensorMapDataType, cuuint32_t, void *, const cuuint64_t *, const cuuint64_t *s, const cuuint32_t *,
                       const cuuint32_t *, CUtensorMapInterleave, CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill) {
    ++asked;
    memcpy(strides, s, sizeof strides);
    return answer;
}
static cudaError_t entry_point(const char *, void **ptr, unsigned long long, cudaDriverEntryPointQueryResult *found) {
    *ptr = reinterpret_cast<void *>(&encode);
    *found = cudaDriverEntryPointSuccess;
    return cudaSuccess;
}
#define cudaGetDriverEntryPoint entry_point
#include "splash_fp8.cuh"
void splash::set_error(const char *, ...) { ++errors; }

int main() {
    alignas(64) CUtensorMap map;
    splash::DecodeParams p;
    memset(&p, 0, sizeof p);
    p.head_end = p.H = 128;
    const long long tib = 1ll << 39;       // elements
    const long long cases[][4] = {         // requests, head stride, request stride, the encoder's answer
        {1, 576, 0, 0}, {1, tib / 64, 0, 0}, {1, tib - 8, -8, 0}, {7, 576, 576 * 128, 0}, {7, 576, tib - 8, 0},
        {7, 576, 0, 0}, {7, 576, -576, 0}, {7, 576, tib, 0}, {1, tib, 0, 0}, {7, 576, 576 * 128, 1}, {1, 576, 0, 1}};
    for (auto &c : cases) {
        asked = errors = 0;
        p.B = (int)c[0]; p.q_stride_head = c[1]; p.q_stride_request = c[2];
        answer = c[3] ? CUDA_ERROR_INVALID_VALUE : CUDA_SUCCESS;
        const bool made = splash::umma::make_query_map(&map, p, 64);
        bool within = true;
        for (int i = 0; asked && i < 3; ++i) within = within && strides[i] % 16 == 0 && strides[i] < (1ull << 40);
        printf("%d%d%d%d ", made, asked, within, errors);
    }
    return 0;
}
"""


def test_no_map_is_no_error(tmp_path):
    src, exe = tmp_path / "map.cu", tmp_path / "map"
    src.write_text(PROGRAM)
    nvcc = os.environ.get("NVCC", "/usr/local/cuda/bin/nvcc")
    subprocess.run([nvcc, "-std=c++17", "-gencode", "arch=compute_100a,code=sm_100a", "-I", build.CSRC, "-o", str(exe), str(src)], check=True)
    got = subprocess.run([str(exe)], capture_output=True, text=True, check=True).stdout.split()
    # made, asked, strides within the encoder's limits, errors
    assert got[:5] == ["1110"] * 5            # a map
    assert got[5:9] == ["0010"] * 4           # none that a map can state: not asked
    assert got[9:] == ["0110"] * 2            # refused
