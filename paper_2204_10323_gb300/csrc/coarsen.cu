// coarsen.cu -- block average of a cell field, the coarsening by which the
// paper builds its 2, 4 and 8 m grids from the 1 m DEM (Methods, "Data").
//
// Output cell (J, I) is the mean of the input cells (j, i) with
// j in [J f, min((J + 1) f, ny)) and i in [I f, min((I + 1) f, nx)): an exact
// f x f block mean where f divides the grid, the mean of the cells present in
// the partial blocks along the far (x = nx, y = ny) edges otherwise.  FP64 sums
// are taken in double; FP32 sums as a float pair where its error is known to be below a hundredth of
// the result's last place, else (and for large factors) in double too.
#include <cuda_runtime.h>

#include <cstdint>
#include <type_traits>

#include "flood_internal.h"

namespace flood {

namespace {

// Factors up to kSmall: one thread per output cell, its rows read as vectors of V elements
// where f and the rows' alignment allow (then a warp reads whole lines, else a row's loads share
// them through L1).  GB300 does two FP64 operations a cycle and SM, so a double add and a
// conversion per input element and a double division per output held 16384^2 by 4 at 1333 us
// (0.86 TB/s); FP32 sums are therefore carried as a float pair (s, c) by Knuth's branch-free two-sum, the
// pair made one of non-overlapping numbers after every row (of blocks above 4 x 4), and the quotient is corrected
// by its remainder: 217 us with the call (5.3 TB/s).
// What the pair can be off by: an addition's error is at most 2^-24 of its result t, and c, their float sum, is rounded
// f times a row (f^2 times a small block), so the additions leave at most f + 1 (f^2) times 2^-48 of the sum m of all
// |t|, the quotient and its correction a few 2^-48 more.  Where that is above 2^-31 of the mean (cells that cancel: about
// one 16 x 16 block in fifty of random signs, none of one sign), or next to either end of the range, or Inf or NaN is
// met, the block is summed in double: 16384^2 of random signs by 4 / 8 / 16 takes 236 / 196 / 430 us, of one sign 217 / 185 / 185.
constexpr int kSmall = 16;

// sum / count, the division of the slow FP64 pipe left out where the quotient is a scaling by a power of two.
__device__ __forceinline__ double mean_of(double sum, int count)
{
    if ((count & (count - 1)) == 0) return sum * __hiloint2double((1023 - (31 - __clz(count))) << 20, 0);
    return sum / (double)count;
}

// The pair (s, c) with |c| at most half a unit in the last place of s.
__device__ __forceinline__ void pair_normalise(float &s, float &c)
{
    const float t = __fadd_rn(s, c), b = __fsub_rn(t, s);
    c = __fadd_rn(__fsub_rn(s, __fsub_rn(t, b)), __fsub_rn(c, b));
    s = t;
}

template <typename T, int V> struct alignas(sizeof(T) * V) Vec {
    T v[V];
};

template <typename T, int V, bool kRows>
__global__ void __launch_bounds__(128) coarsen_small_kernel(const T *__restrict__ src, int nx, int ny, int factor, T *__restrict__ dst,
                                                            int mx, int my)
{
    const int f = !kRows && V == 4 ? 4 : factor;       // (vectors of four and rows of at most four)
    const int I = blockIdx.x * blockDim.x + threadIdx.x;
    if (I >= mx) return;
    const int i0 = I * f, i1 = min(i0 + f, nx);
    for (int J = blockIdx.y; J < my; J += gridDim.y) {
        const int j0 = J * f, j1 = min(j0 + f, ny);
        const int count = (j1 - j0) * (i1 - i0);
        T out;
        double d = 0.0;
        bool whole = true;
        if constexpr (std::is_same<T, float>::value) {
            float s = 0.0f, c = 0.0f, m = 0.0f;
#pragma unroll 4
            for (int j = j0; j < j1; j++) {
                const T *row = src + (size_t)j * nx;
#pragma unroll 2
                for (int i = i0; i < i1; i += V) {      // V divides f and nx: no vector passes the block's end
                    const Vec<T, V> x = *reinterpret_cast<const Vec<T, V> *>(row + i);
#pragma unroll
                    for (int k = 0; k < V; k++) {
                        const float t = __fadd_rn(s, x.v[k]), b = __fsub_rn(t, s);
                        c = __fadd_rn(c, __fadd_rn(__fsub_rn(s, __fsub_rn(t, b)), __fsub_rn(x.v[k], b)));
                        s = t;
                        m = __fadd_rn(m, fabsf(t));
                    }
                }
                if (kRows) pair_normalise(s, c);
            }
            if (!kRows) pair_normalise(s, c);
            const float n = (float)count;
            if ((count & (count - 1)) == 0) {           // a scaling, exact (a sum near zero is not taken)
                out = __fmul_rn(s, __int_as_float((127 - (31 - __clz(count))) << 23));
            } else {
                // the quotient by an approximate reciprocal, its remainder (exact) divided likewise
                const float y = __fdividef(1.0f, n), q = __fmul_rn(s, y);
                out = __fmaf_rn(__fadd_rn(__fmaf_rn(-q, n, s), c), y, q);
            }
            // the error's bound against 2^-31 of the mean, both times 2^31 n
            const bool close = __fmul_rn((float)((kRows ? f : f * f) + 8) * 0x1p-17f, m) <= __fmul_rn(fabsf(out), n);
            whole = isfinite(out) && ((m >= 0x1p-70f && close) || m == 0.0f);
        }
        if (!std::is_same<T, float>::value || !whole) {
            for (int j = j0; j < j1; j++) {
                const T *row = src + (size_t)j * nx;
                for (int i = i0; i < i1; i += V) {
                    const Vec<T, V> x = *reinterpret_cast<const Vec<T, V> *>(row + i);
#pragma unroll
                    for (int k = 0; k < V; k++) d += (double)x.v[k];
                }
            }
            out = (T)mean_of(d, count);
        }
        dst[(size_t)J * mx + I] = out;
    }
}

// Larger factors.
template <typename T>
__global__ void coarsen_kernel(const T *src, int nx, int ny, int f, T *dst, int mx, int my)
{
    const int I = blockIdx.x * blockDim.x + threadIdx.x;
    if (I >= mx) return;
    const int i0 = I * f, i1 = min(i0 + f, nx);
    for (int J = blockIdx.y; J < my; J += gridDim.y) {
        const int j0 = J * f, j1 = min(j0 + f, ny);
        double s = 0.0;
        for (int j = j0; j < j1; j++) {
            const T *row = src + (size_t)j * nx;
            double e = (double)row[i0];                     // row by row: the rounding of 2 f additions, not f^2
            for (int i = i0 + 1; i < i1; i++) e += (double)row[i];
            s = j == j0 ? e : s + e;
        }
        dst[(size_t)J * mx + I] = (T)mean_of(s, (j1 - j0) * (i1 - i0));
    }
}

}  // namespace

template <typename T>
cudaError_t launch_coarsen(const T *src, int nx, int ny, int f, T *dst, cudaStream_t st)
{
    const int mx = (nx + f - 1) / f, my = (ny + f - 1) / f;
    dim3 grid((mx + 127) / 128, my < 65535 ? my : 65535);
    constexpr int V = 16 / sizeof(T);
    const bool small = f <= kSmall;
    const auto run = [&](auto kernel) { kernel<<<grid, 128, 0, st>>>(src, nx, ny, f, dst, mx, my); };
    if (small && f % V == 0 && nx % V == 0 && (uintptr_t)src % 16 == 0)
        run(f > 4 ? coarsen_small_kernel<T, V, true> : coarsen_small_kernel<T, V, false>);
    else if (small && V == 4 && f % 2 == 0 && nx % 2 == 0 && (uintptr_t)src % 8 == 0)
        run(f > 4 ? coarsen_small_kernel<T, 2, true> : coarsen_small_kernel<T, 2, false>);
    else if (small)
        run(f > 4 ? coarsen_small_kernel<T, 1, true> : coarsen_small_kernel<T, 1, false>);
    else
        coarsen_kernel<T><<<grid, 128, 0, st>>>(src, nx, ny, f, dst, mx, my);
    return cudaGetLastError();
}

template cudaError_t launch_coarsen<float>(const float *, int, int, int, float *, cudaStream_t);
template cudaError_t launch_coarsen<double>(const double *, int, int, int, double *, cudaStream_t);

}  // namespace flood
