// copy.cu -- copies between the pitched planes of a handle and dense device arrays
// (flood_read and flood_write_state on device memory).
//
// Bound by HBM: every element is read and written once.  A warp reads and writes
// whole 128-byte lines (512 bytes where both sides allow 16-byte units), eight units
// in flight per thread.  A dense array of nx + 1 columns starts its rows at any
// 4-byte boundary, so those go in single elements.  16384 x 16384 floats: 306 us (7.0
// TB/s), 367 us with 16385 columns (5.9); cudaMemcpy2DAsync took 1056 us for either (2.0).
#include <cuda_runtime.h>

#include <algorithm>
#include <cstdint>

#include "flood_internal.h"
#include "pdl.cuh"

namespace flood {

namespace {

constexpr int kThreads = 256, kUnroll = 8;

// rows x cols units of type U; pitches in units.  A block has kThreads / tx rows of tx threads.
template <typename U>
__global__ void __launch_bounds__(kThreads)
    copy_rows_kernel(U *__restrict__ dst, size_t dpitch, const U *__restrict__ src, size_t spitch, size_t cols, size_t rows)
{
    pdl_wait();
    pdl_launch();
    const size_t tx = blockDim.x;
    for (size_t r = (size_t)blockIdx.x * blockDim.y + threadIdx.y; r < rows; r += (size_t)gridDim.x * blockDim.y) {
        const U *s = src + r * spitch;
        U *d = dst + r * dpitch;
        size_t c = threadIdx.x;
        for (; c + (kUnroll - 1) * tx < cols; c += kUnroll * tx) {
            U v[kUnroll];
#pragma unroll
            for (int k = 0; k < kUnroll; k++) v[k] = __ldcs(s + c + k * tx);
#pragma unroll
            for (int k = 0; k < kUnroll; k++) __stcs(d + c + k * tx, v[k]);
        }
        for (; c < cols; c += tx) __stcs(d + c, __ldcs(s + c));
    }
}

template <typename U>
cudaError_t launch(void *dst, size_t dpitch, const void *src, size_t spitch, size_t width, size_t rows, cudaStream_t st)
{
    const size_t cols = width / sizeof(U);
    int tx = 32;                                   // a row's threads: one batch of a short row, all of them for a long one
    while (tx < kThreads && (size_t)tx * kUnroll < cols) tx *= 2;
    const int ty = kThreads / tx;
    const size_t blocks = (rows + ty - 1) / ty;
    return launch_pdl(copy_rows_kernel<U>, (unsigned)std::min<size_t>(blocks, 1u << 20), dim3(tx, ty), st, (U *)dst,
                      dpitch / sizeof(U), (const U *)src, spitch / sizeof(U), cols, rows);
}

// Copy blockIdx.y of the list.
__global__ void __launch_bounds__(kThreads) halo_rows_kernel(const HaloRows *__restrict__ copies)
{
    const HaloRows c = copies[blockIdx.y];
    for (int64_t k = (int64_t)blockIdx.x * kThreads + threadIdx.x; k < c.units; k += (int64_t)gridDim.x * kThreads)
        reinterpret_cast<float4 *>(c.dst)[k] = reinterpret_cast<const float4 *>(c.src)[k];
}

}  // namespace

cudaError_t launch_halo_rows(const HaloRows *copies, int n, int64_t max_units, cudaStream_t st)
{
    if (n <= 0 || max_units <= 0) return cudaSuccess;
    const int blocks = (int)std::min<int64_t>((max_units + kThreads - 1) / kThreads, 64);
    for (int k = 0; k < n; k += 65535)
        halo_rows_kernel<<<dim3(blocks, std::min(n - k, 65535)), kThreads, 0, st>>>(copies + k);
    return cudaGetLastError();
}

cudaError_t launch_copy_rows(void *dst, size_t dpitch, const void *src, size_t spitch, size_t width, size_t rows,
                             cudaStream_t st)
{
    if (width == 0 || rows == 0) return cudaSuccess;
    const size_t any = (size_t)(uintptr_t)dst | (size_t)(uintptr_t)src | dpitch | spitch | width;
    if (any % 16 == 0) return launch<float4>(dst, dpitch, src, spitch, width, rows, st);
    if (any % 8 == 0) return launch<double>(dst, dpitch, src, spitch, width, rows, st);
    if (any % 4 == 0) return launch<float>(dst, dpitch, src, spitch, width, rows, st);
    return cudaMemcpy2DAsync(dst, dpitch, src, spitch, width, rows, cudaMemcpyDeviceToDevice, st);
}

}  // namespace flood
