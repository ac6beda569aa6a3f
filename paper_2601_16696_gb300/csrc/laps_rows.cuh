// laps_rows.cuh -- kernels that copy or add rows of floats between the caller's [M][d]
// arrays and the padded ones: an element of the row-major array, index k = row w + column,
// at a time, consecutive lanes on consecutive k, so that few long rows, many short ones and
// everything between spread over the GPU alike.
#pragma once
#include <cuda_runtime.h>

#include <cstdint>

namespace laps {

// k -> (row, column) by a multiplication and a shift (Granlund and Montgomery, "Division
// by invariant integers using multiplication", PLDI 1994): for k < 2^31 and w >= 1,
// k / w = k m >> (31 + s) with s = ceil(log2 w), m = ceil(2^(31 + s) / w) < 2^32.
struct RowIndex {
    int64_t n;    // elements
    uint32_t w;   // row length
    uint32_t m;
    int s;        // 31 + ceil(log2 w)
};
inline RowIndex row_index(int64_t M, int w) {
    RowIndex r{M * w, (uint32_t)w, 0, 31};
    while ((1u << (r.s - 31)) < r.w) ++r.s;
    r.m = (uint32_t)(((1ull << r.s) + r.w - 1) / r.w);
    return r;
}
// Blocks of 256 threads: at most about one wave (eight an SM), whose threads then take
// several elements, four in flight, rather than a second wave of blocks.
inline int row_blocks(const RowIndex& r) { return (int)(r.n < 256 * 1216 ? (r.n + 255) / 256 : 1216); }

__host__ __device__ __forceinline__ void row_of(const RowIndex& r, uint32_t k, uint32_t& row, int& col) {
    row = (uint32_t)(((uint64_t)k * r.m) >> r.s);
    col = (int)(k - row * r.w);
}
__host__ __device__ __forceinline__ void row_of(const RowIndex& r, uint64_t k, uint64_t& row, int& col) {
    row = k / r.w;
    col = (int)(k - row * r.w);
}
// store(v, k, row, column) of v = load(row, column) for the elements of this thread
template <typename I, class L, class S>
__device__ __forceinline__ void for_elements_as(const RowIndex& r, L load, S store) {
    const I n = (I)r.n, step = (I)(gridDim.x * blockDim.x);
    for (I k0 = (I)(blockIdx.x * blockDim.x + threadIdx.x); k0 < n; k0 += 4 * step) {
        I row[4];
        int col[4];
        float v[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            const I k = k0 + u * step;
            if (k >= n) break;
            row_of(r, k, row[u], col[u]);
            v[u] = load((int64_t)row[u], col[u]);
        }
#pragma unroll
        for (int u = 0; u < 4; ++u)
            if (k0 + u * step < n) store(v[u], (int64_t)(k0 + u * step), (int64_t)row[u], col[u]);
    }
}
template <class L, class S>
__device__ __forceinline__ void for_elements(const RowIndex& r, L load, S store) {
    if (r.n <= 0x7fffffff) for_elements_as<uint32_t>(r, load, store);
    else for_elements_as<uint64_t>(r, load, store);
}
// Rows of d_pad floats to rows of r.w (times scale, if any).  Measured, us a launch (a 64-bit
// division an element and one load in flight; a warp a row; this): M = 16384, d = 100 8.3,
// 4.7, 4.7; M = 65536, d = 10 5.3, 9.2, 3.5; M = 2, d = 10^4 2.4, 35, 2.4; M = 4096,
// d = 10^4 (328 MB) 111, 107, 76.
__device__ __forceinline__ void unpack_rows(const float* __restrict__ src, const float* __restrict__ scale,
                                            float* __restrict__ dst, const RowIndex& r, int d_pad) {
    for_elements(
        r, [&](int64_t row, int col) { return src[row * d_pad + col] * (scale ? scale[col] : 1.0f); },
        [&](float v, int64_t k, int64_t, int) { dst[k] = v; });
}

}  // namespace laps
