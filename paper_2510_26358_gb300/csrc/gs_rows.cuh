// Copies of splat rows into a compacted array, for the kernels that keep,
// move, split or create splats (lifecycle, partition).  A block owns a chunk of
// kRowChunk input rows, whose output rows are consecutive; `rows` (shared)
// names the input row of each, relative to the chunk, so the copy runs over the
// output's elements: consecutive threads write consecutive words, in 16-byte
// pieces where the row and the arrays allow it, four in flight a thread.
// Bound by memory; against a warp a row (48 words in two uneven turns, one
// row after the other) the lifecycle pass of 1M splats with moments went from
// 878 to 252 us (of 209 at the copy rate), the offload of 100k of 500k splats
// to pinned host memory from 325 to 160 us (25 MB over the link to the host).
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

namespace gs {

constexpr int kRowChunk = 512;
// what an entry of `rows` holds besides the input row (9 bits)
constexpr uint32_t kRowIndex = kRowChunk - 1, kRowChild = 0x400, kRowSplit = 0x800, kRowReset = 0x1000,
                   kRowFresh = 0x8000;
enum RowMode { ROWS_COPY, ROWS_ZERO_FRESH, ROWS_SKIP_SPLIT };

// n output rows of W elements: out[r][:] = in[rows[r] & kRowIndex][:]
template <int NT, int W, RowMode MODE, typename E>
__device__ __forceinline__ void copy_elements(const E *__restrict__ in, E *__restrict__ out, const uint16_t *rows,
                                              int n) {
    constexpr int U = 4;
    const int total = n * W;
    for (int i0 = threadIdx.x; i0 < total; i0 += U * NT) {
        E v[U];
        bool write[U];
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const int i = i0 + u * NT;
            write[u] = i < total;
            v[u] = E{};
            if (!write[u]) continue;
            const int r = i / W, c = i - r * W;
            const uint32_t s = rows[r];
            if (MODE == ROWS_SKIP_SPLIT && (s & kRowSplit)) write[u] = false;
            else if (!(MODE == ROWS_ZERO_FRESH && (s & kRowFresh))) v[u] = in[(s & kRowIndex) * W + c];
        }
#pragma unroll
        for (int u = 0; u < U; ++u)
            if (write[u]) out[i0 + u * NT] = v[u];
    }
}

// The same for floats, in 16-byte pieces when W is a multiple of four and
// both arrays start on 16-byte boundaries.
template <int NT, int W, RowMode MODE>
__device__ __forceinline__ void copy_rows(const float *in, float *out, const uint16_t *rows, int n) {
    if constexpr (W % 4 == 0) {
        if ((((uintptr_t)in | (uintptr_t)out) & 15) == 0) {
            copy_elements<NT, W / 4, MODE>(reinterpret_cast<const float4 *>(in), reinterpret_cast<float4 *>(out), rows, n);
            return;
        }
    }
    copy_elements<NT, W, MODE>(in, out, rows, n);
}

}  // namespace gs
