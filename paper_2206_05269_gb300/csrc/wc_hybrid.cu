// The reduce of the paper's hybrid pipeline (Sec. 3.3 "Reduce on GPU",
// measured in Sec. 4.1): the host has mapped every document to a dictionary
// and laid the per-document counts of each word out as one row of a
// zero-padded matrix; the GPU sums each row.  It reads the matrix once: bound by
// HBM (rows x cols x 4 bytes read, rows x 8 written).  One warp sums one row, a
// shuffle reduction at its end.
//   Rows of more than kNarrowCols: 16-byte loads (the row's first and last words
// that are not part of an aligned 16 bytes by single loads), eight a lane issued
// before the first sum, so a row of 1,000 counts is in flight at once; one block
// for every eight rows, which evens out the rows better than a grid of resident
// blocks.
//   Narrower rows: 4-byte loads, four a lane in flight, and resident blocks that
// take rows in turn: such a row is a few loads, and the eight 16-byte ones with
// their bounds were most of its time.
// us, 4-byte | 16-byte: 30,000 rows of 100 10.9 | 15.0, of 400 19.1 | 17.1, of 512
// 21.1 | 19.1, of 1,000 39.6 | 27.3; 300,000 rows of 31 41.6 | 94.9, of 256 70 | 95, of
// 400 101 | 101, of 512 117 | 122, of 640 140 | 130, of 1,000 222 | 179.
#include <cuda_runtime.h>

#include <cstdint>

#include "wc_internal.h"

namespace wc {

__device__ __forceinline__ uint4 ld_once16(const uint4 *p) {
    uint4 v;
    asm volatile("ld.global.nc.L1::no_allocate.v4.u32 {%0, %1, %2, %3}, [%4];"
                 : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w)
                 : "l"(p));
    return v;
}

constexpr unsigned long long kNarrowCols = 512;
constexpr int kRowLoads = 8;  // 16-byte loads a lane has in flight
__global__ void __launch_bounds__(256) k_row_sums(const uint32_t *m, unsigned long long rows, unsigned long long cols,
                                                  unsigned long long *out) {
    const uint32_t lane = threadIdx.x & 31u;
    const unsigned long long nw = ((unsigned long long)gridDim.x * blockDim.x) >> 5;
    for (unsigned long long r = ((unsigned long long)blockIdx.x * blockDim.x + threadIdx.x) >> 5; r < rows; r += nw) {
        const uint32_t *row = m + r * cols;
        // row[0, head) up to the first 16-byte boundary, nv aligned groups of four, the rest
        unsigned long long head = (4u - (uint32_t)(reinterpret_cast<uintptr_t>(row) >> 2)) & 3u;
        if (head > cols) head = cols;
        const unsigned long long nv = (cols - head) >> 2, tail = head + 4 * nv;
        const uint4 *v = reinterpret_cast<const uint4 *>(row + head);
        unsigned long long s = 0;
        for (unsigned long long b = 0; b < nv; b += 32 * kRowLoads) {
            uint4 x[kRowLoads];
#pragma unroll
            for (int q = 0; q < kRowLoads; q++) {
                const unsigned long long i = b + 32u * q + lane;
                x[q] = i < nv ? ld_once16(v + i) : make_uint4(0u, 0u, 0u, 0u);
            }
#pragma unroll
            for (int q = 0; q < kRowLoads; q++)
                s += ((unsigned long long)x[q].x + x[q].y) + ((unsigned long long)x[q].z + x[q].w);
        }
        if (lane < head) s += __ldg(row + lane);
        if (tail + lane < cols) s += __ldg(row + tail + lane);
        for (int o = 16; o; o >>= 1) s += __shfl_xor_sync(0xFFFFFFFFu, s, o);
        if (lane == 0) out[r] = s;
    }
}

__global__ void __launch_bounds__(256) k_row_sums_narrow(const uint32_t *m, unsigned long long rows,
                                                         unsigned long long cols, unsigned long long *out) {
    const uint32_t lane = threadIdx.x & 31u;
    const unsigned long long nw = ((unsigned long long)gridDim.x * blockDim.x) >> 5;
    for (unsigned long long r = ((unsigned long long)blockIdx.x * blockDim.x + threadIdx.x) >> 5; r < rows; r += nw) {
        const uint32_t *row = m + r * cols;
        unsigned long long s = 0, c = lane;
        for (; c + 96 < cols; c += 128)
            s += (unsigned long long)__ldg(row + c) + __ldg(row + c + 32) + __ldg(row + c + 64) + __ldg(row + c + 96);
        for (; c < cols; c += 32) s += __ldg(row + c);
        for (int o = 16; o; o >>= 1) s += __shfl_xor_sync(0xFFFFFFFFu, s, o);
        if (lane == 0) out[r] = s;
    }
}

cudaError_t launch_row_sums(const uint32_t *m, unsigned long long rows, unsigned long long cols,
                            unsigned long long *out, cudaStream_t s) {
    if (!rows) return cudaSuccess;
    if (cols <= kNarrowCols) {
        int dev = 0, sms = 1;
        cudaGetDevice(&dev);
        cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
        const unsigned long long blocks = (rows + 7) / 8, resident = (unsigned long long)(sms > 0 ? sms : 1) * 16;
        k_row_sums_narrow<<<(unsigned)(blocks < resident ? blocks : resident), 256, 0, s>>>(m, rows, cols, out);
        return cudaGetLastError();
    }
    const unsigned long long want = (rows + 7) / 8, cap = 1ull << 20;  // 8 warps (rows) a block
    k_row_sums<<<(unsigned)(want < cap ? want : cap), 256, 0, s>>>(m, rows, cols, out);
    return cudaGetLastError();
}

}  // namespace wc
