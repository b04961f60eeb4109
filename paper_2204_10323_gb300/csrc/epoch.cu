// epoch.cu -- per-epoch and bookkeeping kernels: the time-step rule, the
// Eq. 6 inflow distribution, and deterministic reductions (h_max, volume,
// gauge gathers).
#include <cfloat>

#include "device_common.cuh"
#include "pdl.cuh"

namespace flood {

namespace {

// Time-step rule at an epoch start: constant, frozen (adjoint replays), or
// dt = min(dt_cap, alpha dx / sqrt(g h_max)); h_max = 0 gives dt_cap.
__device__ double epoch_dt(const Geom &G, double hmax, const double *fixed_dt)
{
    if (fixed_dt) return *fixed_dt;
    if (G.dt_mode == 1) return G.dt_const;
    if (!(hmax > 0.0)) return G.dt_cap;
    return fmin(G.dt_cap, G.cfl_alpha * G.dx / sqrt(G.g * hmax));
}

__device__ void epoch_begin_body(const Geom &G, Ctrl *ctrl, double *t_list, int E, const double *fixed_dt)
{
    double hmax = __longlong_as_double((long long)ctrl->hmax_bits);
    if (!isfinite(hmax)) ctrl->status |= kStatusNonfinite;
    // the epoch that just ended: its dt against the Courant limit of the depth it ended with (not for
    // replays of a logged schedule, whose control block is restored after them)
    if (!fixed_dt && ctrl->dt > 0.0 && hmax > 0.0 && ctrl->dt * sqrt(G.g * hmax) > G.dx) {
        ctrl->cfl_exceed += 1.0;
        ctrl->status |= kStatusCfl;
    }
    const double dt = epoch_dt(G, hmax, fixed_dt);
    ctrl->dt = dt;
    ctrl->h_max = hmax;
    ctrl->hmax_bits = 0ull;
    double t = ctrl->t;
    t_list[0] = t;
    for (int s = 0; s < E; s++) {
        t = t + dt;
        t_list[s + 1] = t;
    }
}

__global__ void epoch_begin_kernel(Geom G, Ctrl *ctrl, double *t_list, int E, const double *fixed_dt)
{
    if (threadIdx.x != 0 || blockIdx.x != 0) return;
    epoch_begin_body(G, ctrl, t_list, E, fixed_dt);
}

// One thread per simulation of a batch.
template <typename T>
__global__ void epoch_begin_batched_kernel(const EpochArgs<T> *tab, int n, int E)
{
    const int k = blockIdx.x * blockDim.x + threadIdx.x;
    if (k >= n) return;
    epoch_begin_body(tab[k].geo, tab[k].ctrl, tab[k].t_list, E, nullptr);
}

// Linear interpolation in the hydrograph table, constant past both ends.
__device__ double hydrograph(const double *ts, const double *qs, int n, double t)
{
    if (n <= 0) return 0.0;
    if (t <= ts[0]) return qs[0];
    for (int k = 1; k < n; k++)
        if (t <= ts[k]) {
            double w = (t - ts[k - 1]) / (ts[k] - ts[k - 1]);
            return qs[k - 1] + w * (qs[k] - qs[k - 1]);
        }
    return qs[n - 1];
}

// Eq. 5 discharge of one cell (m^3/s) at depth hh.
__device__ __forceinline__ double manning_cell(double hh, double sqrtS, double n, double dx, int form)
{
    if (form == 0) return dx * pow(hh, 5.0 / 3.0) * sqrtS / n;
    return dx * dx * pow(hh, 2.0 / 3.0) * sqrtS / n;
}

// FP32 handles evaluate Eq. 5 in single precision inside the solve (the
// final rescale makes the section total exact either way); FP64 handles keep
// the double-precision evaluation of the plain definition.
__device__ __forceinline__ double manning_cell_t(double hh, double sqrtS, float n, double dx, int form)
{
    float h = (float)hh, p = form == 0 ? 5.0f / 3.0f : 2.0f / 3.0f;
    float a = form == 0 ? (float)dx : (float)(dx * dx);
    return (double)(a * powf(h, p) * (float)sqrtS / n);
}

__device__ __forceinline__ double manning_cell_t(double hh, double sqrtS, double n, double dx, int form)
{
    return manning_cell(hh, sqrtS, n, dx, form);
}

constexpr int kInflowThreads = 128;

// Sections of at most this many cells are solved by warp 0 alone: a search
// step then costs one warp reduction instead of two block barriers, and the
// solve is latency-bound (the sections of the workloads hold 12-512 cells).
// FP64 handles evaluate Eq. 5 with the slow double pow, so only the smallest
// sections go to one warp there.  The choice depends on the section alone, so
// a single grid and an ensemble member solve a section in the same order.
constexpr int kWarpCells = 1024;     // shared-memory copy of a one-warp section's z and n

template <typename T>
__device__ __forceinline__ bool one_warp(const InflowSec &S)
{
    return S.ncell <= (sizeof(T) == 4 ? kWarpCells : 32);
}

// Depth exponent of Eq. 5.
__device__ __forceinline__ double depth_exponent(int form) { return form == 0 ? 5.0 / 3.0 : 2.0 / 3.0; }

// Sum of a one-warp section's Eq. 5 discharges at level W from its cells' z
// and n staged in shared memory, and its slope (every lane of warp 0 gets them).
template <typename T>
__device__ double section_total_warp(const InflowSec &S, const T *sz, const T *sn, double W, double dx,
                                     int form, double &slope)
{
    double s = 0.0, d = 0.0;
    for (int c = threadIdx.x; c < S.ncell; c += 32) {
        double hh = W - (double)sz[c];
        if (hh > 0.0) {
            const double w = manning_cell_t(hh, S.sqrtS, sn[c], dx, form);
            s += w;
            d += depth_exponent(form) * w / hh;
        }
    }
    slope = warp_sum(d);
    return warp_sum(s);
}

// The level search.  The section's discharge is increasing in the level W and, for the cross-section form
// (h^(5/3)), convex: Newton's method from above falls monotonically to the root in a handful of evaluations (in double
// and on one warp in single precision; 26 on longer single-precision sections), where the halvings took 25 (FP32, one
// warp) or 41 and more, each a chain of powers and a sum over the section.
// An iteration that leaves the bracket is replaced by a halving, as are all of them for the literal form
// (h^(2/3): its slope is infinite where a cell falls dry).

// x moved n floats up (down for n < 0).
__device__ __forceinline__ float float_step(float x, int n)
{
    int i = __float_as_int(x);
    i = i < 0 ? (int)(0x80000000u - (unsigned)i) : i;  // floats in order as integers
    i += n;
    return __int_as_float(i < 0 ? (int)(0x80000000u - (unsigned)i) : i);
}

// FP32 handles, one-warp sections: Eq. 6 in single precision throughout the search (the level W, Eq. 5
// per cell, the warp's butterfly sum), to neighbouring floats lo, hi with total(lo) < Q <= total(hi): W = hi;
// then each cell's discharge rescaled to Q_in in double.  An epoch start of 16 steps of a 13-cell section: 17 us
// in two launches with the halvings, 10.4 in one with Newton's steps; FP64 179 and 55.5 us.
__device__ void inflow_solve_warp_f32(const InflowSec &S, const float *sz, const float *sn, float zmin, double Q,
                                      double dx, int form, float *out, double *W_slot)
{
    const int lane = threadIdx.x;
    const float p = form == 0 ? 5.0f / 3.0f : 2.0f / 3.0f;
    const float a = form == 0 ? (float)dx : (float)(dx * dx);
    const float sq = (float)S.sqrtS;
    // the discharge at level W, and its slope in d
    auto total = [&](float W, float &d) {
        float s = 0.0f;
        d = 0.0f;
        for (int c = lane; c < S.ncell; c += 32) {
            const float hh = W - sz[c];
            if (hh > 0.0f) {
                const float w = a * powf(hh, p) * sq / sn[c];
                s += w;
                d += __fdividef(p * w, hh);
            }
        }
        for (int o = 16; o > 0; o >>= 1) {
            s += __shfl_xor_sync(0xffffffffu, s, o);
            d += __shfl_xor_sync(0xffffffffu, d, o);
        }
        return s;
    };
    const float Qf = (float)Q;
    float Hb = 1.0f, d, f = total(zmin + Hb, d);
    while (f < Qf && Hb < 1e12f) {
        Hb *= 2.0f;
        f = total(zmin + Hb, d);
    }
    float lo = zmin, hi = zmin + Hb;                   // f, d: at hi
    int step = 1;                                      // floats to move when Newton's step is lost in rounding
    for (int it = 0; it < 200; it++) {
        const float half = 0.5f * (lo + hi);
        if (!(half > lo && half < hi)) break;          // neighbouring floats
        float W = half;
        if (form == 0) {
            W = hi - __fdividef(f - Qf, d);
            if (!(W > lo && W < hi)) {
                // at the root up to rounding: a few floats above lo, or below hi
                W = W <= lo ? float_step(lo, step) : float_step(hi, -step);
                step *= 2;
                if (!(W > lo && W < hi)) W = half;
            }
        }
        float dW;
        const float fW = total(W, dW);
        if (fW < Qf) lo = W;
        else {
            hi = W;
            f = fW;
            d = dW;
        }
    }
    const float W = hi;
    if (lane == 0 && W_slot) *W_slot = (double)W;
    const double tot = (double)total(W, d);
    for (int c = lane; c < S.ncell; c += 32) {
        const float hh = W - sz[c];
        const float w = hh > 0.0f ? a * powf(hh, p) * sq / sn[c] : 0.0f;
        out[c] = (float)(((double)w * (Q / tot)) / dx);
    }
}

// The depth above zmin at which a one-warp section carries about Q, in single precision (form 0).
template <typename T>
__device__ float level_guess_f32(const InflowSec &S, const T *sz, const T *sn, double zmin, double Q, double dx)
{
    const float a = (float)(dx * S.sqrtS), Qf = (float)Q;
    auto total = [&](float H, float &d) {
        float s = 0.0f;
        d = 0.0f;
        for (int c = threadIdx.x; c < S.ncell; c += 32) {
            const float hh = H - (float)((double)sz[c] - zmin);
            if (hh > 0.0f) {
                const float w = __fdividef(a * __powf(hh, 5.0f / 3.0f), (float)sn[c]);
                s += w;
                d += __fdividef(5.0f / 3.0f * w, hh);
            }
        }
        for (int o = 16; o > 0; o >>= 1) {
            s += __shfl_xor_sync(0xffffffffu, s, o);
            d += __shfl_xor_sync(0xffffffffu, d, o);
        }
        return s;
    };
    float H = 1.0f, d, f = total(H, d);
    while (f < Qf && H < 1e12f) {
        H *= 2.0f;
        f = total(H, d);
    }
    for (int it = 0; it < 12; it++) {
        const float step = __fdividef(f - Qf, d);
        if (!(step > 1e-6f * H)) break;
        H -= step;
        f = total(H, d);
    }
    return H;
}

// Block-wide sum of the section's Eq. 5 discharges at level W, and its slope (all threads get them).
template <typename T>
__device__ double section_total(const InflowSec &S, const int64_t *cells, const T *z, const T *n,
                                double W, double dx, int form, double *red, double &slope)
{
    double s = 0.0, d = 0.0;
    for (int c = threadIdx.x; c < S.ncell; c += kInflowThreads) {
        int64_t idx = cells[S.cell0 + c];
        double hh = W - (double)z[idx];
        if (hh > 0.0) {
            const double w = manning_cell_t(hh, S.sqrtS, n[idx], dx, form);
            s += w;
            d += depth_exponent(form) * w / hh;
        }
    }
    s = warp_sum(s);
    d = warp_sum(d);
    __syncthreads();
    if ((threadIdx.x & 31) == 0) {
        red[threadIdx.x >> 5] = s;
        red[kInflowThreads / 32 + (threadIdx.x >> 5)] = d;
    }
    __syncthreads();
    double t = 0.0;
    slope = 0.0;
    for (int w = 0; w < kInflowThreads / 32; w++) {
        t += red[w];
        slope += red[kInflowThreads / 32 + w];
    }
    return t;
}

// Eq. 6 for (step s of the epoch, inflow section k), by warp 0 or the whole
// block (one_warp): the level W with sum_c Q_c(W) = Q_in(t) bracketed on [min z, min z + H]
// (H doubled from 1 m), 200 steps at most or a bracket below 1e-12 m, W = upper end; then
// each cell's discharge scaled by Q_in / sum, stored as unit-width flux.
template <typename T>
__device__ void inflow_body(const Geom &G, const InflowSec *secs, int nsec, const int64_t *cells,
                            const double *tab_t, const double *tab_q, const T *z, const T *n,
                            const double t, T *inflow_q, int n_slots, double *inflow_Q, double *W_out,
                            const int s, const int k, double *red, T *sz, T *sn)
{
    const int tid = threadIdx.x;
    const InflowSec S = secs[k];
    const double Q = hydrograph(tab_t + S.tab0, tab_q + S.tab0, S.ntab, t);
    T *out = inflow_q + (size_t)s * n_slots + S.slot0;
    // a section that covers no cell carries no discharge
    if (tid == 0) inflow_Q[(size_t)s * nsec + k] = S.ncell > 0 ? Q : 0.0;
    double zmin = DBL_MAX;
    for (int c = tid; c < S.ncell; c += kInflowThreads) zmin = fmin(zmin, (double)z[cells[S.cell0 + c]]);
    for (int o = 16; o > 0; o >>= 1) zmin = fmin(zmin, __shfl_xor_sync(0xffffffffu, zmin, o));
    if ((tid & 31) == 0) red[tid >> 5] = zmin;
    __syncthreads();
    for (int w = 0; w < kInflowThreads / 32; w++) zmin = fmin(zmin, red[w]);
    if (!(Q > 0.0) || S.ncell == 0) {
        for (int c = tid; c < S.ncell; c += kInflowThreads) out[c] = T(0);
        return;
    }
    const bool warp_only = one_warp<T>(S);
    if (warp_only && tid >= 32) return;           // warp 0 solves and distributes
    const int nthreads = warp_only ? 32 : kInflowThreads;
    const double dx = G.dx;
    const int form = G.bc_form;
    if (warp_only) {                              // the section's z and n, read once
        for (int c = tid; c < S.ncell; c += 32) {
            const int64_t idx = cells[S.cell0 + c];
            sz[c] = z[idx];
            sn[c] = n[idx];
        }
        __syncwarp();
        if constexpr (sizeof(T) == 4) {
            inflow_solve_warp_f32(S, sz, sn, (float)zmin, Q, dx, form, out,
                                  W_out ? W_out + (size_t)s * nsec + k : nullptr);
            return;
        }
    }
    auto total_at = [&](double W, double &d) {
        return warp_only ? section_total_warp(S, sz, sn, W, dx, form, d)
                         : section_total(S, cells, z, n, W, dx, form, red, d);
    };
    // FP64, one warp: the level in single precision first (depths above the lowest bed, so that high ground
    // costs no digits), and the double search from just above it: three or four evaluations of the slow FP64
    // powers instead of ten
    double hi = 0.0, d = 0.0, f = -1.0;
    if (sizeof(T) == 8 && warp_only && form == 0) {
        const float H = level_guess_f32(S, sz, sn, zmin, Q, dx);
        hi = zmin + (double)H * (1.0 + 1e-5);
        f = total_at(hi, d);
    }
    if (!(f >= Q && f < 1e300)) {
        double Hb = 1.0;
        f = total_at(zmin + Hb, d);
        while (f < Q && Hb < 1e12) {
            Hb *= 2.0;
            f = total_at(zmin + Hb, d);
        }
        hi = zmin + Hb;
    }
    double lo = zmin;                                  // f, d: at hi
    // What the section's sum resolves: in double a few roundings of the level, in single precision (sections beyond a
    // warp's cells) those of the depths.  Newton's step keeps that far from the bracket's ends (twice as far each time it
    // has to, as the sum's own rounding may hide the root), so that the bracket closes on the root from both sides.  (Ends
    // 0.9e-12 m apart, the bracket's width, left the level up to that far above in double, and crept along the steps of a
    // single-precision sum: 75 to 110 evaluations where the halvings take 43; now 26.)
    double least = 1.0;
    for (int it = 0; it < 200 && hi - lo >= 1e-12; it++) {
        const double half = 0.5 * (lo + hi);
        if (!(half > lo && half < hi)) break;          // neighbouring doubles
        double W = half;
        const double r = least * (sizeof(T) == 8 ? 0x1p-51 * fmax(fabs(hi), hi - zmin) : 0x1p-22 * (hi - zmin));
        if (form == 0 && it < 60 && hi - lo > 4.0 * r) {
            W = hi - (f - Q) / d;
            if (W > hi - r || W < lo + r) {
                W = W > hi - r ? hi - r : lo + r;
                least *= 2.0;
            }
            if (!(W > lo && W < hi)) W = half;
        }
        double dW;
        const double fW = total_at(W, dW);
        if (fW < Q) lo = W;
        else {
            hi = W;
            f = fW;
            d = dW;
        }
    }
    const double W = hi;
    if (tid == 0 && W_out) W_out[(size_t)s * nsec + k] = W;
    const double total = f;                            // at W
    for (int c = tid; c < S.ncell; c += nthreads) {
        int64_t idx = cells[S.cell0 + c];
        double hh = W - (double)z[idx];
        double w = hh > 0.0 ? manning_cell_t(hh, S.sqrtS, n[idx], dx, form) : 0.0;
        out[c] = T((w * (Q / total)) / dx);
    }
}

// An epoch start in the blocks of its inflow solve, in place of a launch of its own (one thread's few
// microseconds and a launch gap): each block derives the time step and its step's start time for itself,
// and the last of the simulation's `blocks` blocks to have read the control block writes the epoch's into it.
__device__ double epoch_time(const Geom &G, const Ctrl *ctrl, const double *fixed_dt, int s, double *shared_t)
{
    if (threadIdx.x == 0) {
        const double dt = epoch_dt(G, __longlong_as_double((long long)ctrl->hmax_bits), fixed_dt);
        double t = ctrl->t;
        for (int k = 0; k < s; k++) t = t + dt;        // the additions of t_list
        *shared_t = t;
    }
    __syncthreads();
    return *shared_t;
}

// By the block's last thread, which a one-warp solve leaves free.
__device__ void epoch_commit(const Geom &G, Ctrl *ctrl, double *t_list, int E, const double *fixed_dt, unsigned blocks)
{
    if (threadIdx.x != kInflowThreads - 1) return;
    __threadfence();
    if (atomicAdd(&ctrl->epoch_blocks, 1u) != blocks - 1) return;
    __threadfence();
    ctrl->epoch_blocks = 0;
    epoch_begin_body(G, ctrl, t_list, E, fixed_dt);
}

// Eq. 6 for (step, section) = block (x, y); kBegin: the epoch starts here (ctrl, fixed_dt), else t_list holds
// its times.
template <typename T, bool kBegin>
__global__ void __launch_bounds__(kInflowThreads)
    inflow_kernel(Geom G, Ctrl *ctrl, const double *fixed_dt, const InflowSec *secs, int nsec, const int64_t *cells,
                  const double *tab_t, const double *tab_q, const T *z, const T *n, double *t_list, int E, T *inflow_q,
                  int n_slots, double *inflow_Q, double *W_out)
{
    __shared__ double red[2 * kInflowThreads / 32], st;
    __shared__ T sz[kWarpCells], sn[kWarpCells];
    pdl_wait();
    pdl_launch();
    const double t = kBegin ? epoch_time(G, ctrl, fixed_dt, blockIdx.x, &st) : t_list[blockIdx.x];
    inflow_body<T>(G, secs, nsec, cells, tab_t, tab_q, z, n, t, inflow_q, n_slots, inflow_Q, W_out, blockIdx.x,
                   blockIdx.y, red, sz, sn);
    if (kBegin) epoch_commit(G, ctrl, t_list, E, fixed_dt, gridDim.x * gridDim.y);
}

// The same for every (step, section) of a batch of simulations: block (s, task).
template <typename T, bool kBegin>
__global__ void __launch_bounds__(kInflowThreads) inflow_batched_kernel(const EpochArgs<T> *tab, const int2 *tasks)
{
    __shared__ double red[2 * kInflowThreads / 32], st;
    __shared__ T sz[kWarpCells], sn[kWarpCells];
    const int2 task = tasks[blockIdx.y];
    const EpochArgs<T> &A = tab[task.x];
    const double t = kBegin ? epoch_time(A.geo, A.ctrl, nullptr, blockIdx.x, &st) : A.t_list[blockIdx.x];
    inflow_body<T>(A.geo, A.secs, A.nsec, A.cells, A.tab_t, A.tab_q, A.z, A.n, t, A.inflow_q, A.n_slots,
                   A.inflow_Q, A.inflow_W, blockIdx.x, task.y, red, sz, sn);
    if (kBegin) epoch_commit(A.geo, A.ctrl, A.t_list, gridDim.x, nullptr, gridDim.x * A.nsec);
}

// A thread's share of the depths, in 16-byte vectors along the rows (they start on 128-byte boundaries), two rows
// in flight: fn(value) per depth.  Rows over the blocks' warps, vectors over lanes.  One element at a time, a row
// per block, the depth maximum of 1024^2 took 11.8 us.
template <typename T, typename Fn>
__device__ __forceinline__ void for_depths(const Geom &G, const T *h, Fn fn)
{
    constexpr int V = 16 / sizeof(T);
    struct alignas(16) Vec {
        T v[V];
    };
    const int lane = threadIdx.x & 31, warps = gridDim.x * (blockDim.x >> 5);
    const int whole = G.nx / V;                        // whole vectors of a row
    for (int j = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5); j < G.ny; j += warps) {
        const T *row = h + (size_t)j * G.pitch;
        int i = lane;
        for (; i + 96 < whole; i += 128) {
            Vec x[4];
#pragma unroll
            for (int u = 0; u < 4; u++) x[u] = reinterpret_cast<const Vec *>(row)[i + 32 * u];
#pragma unroll
            for (int u = 0; u < 4; u++)
#pragma unroll
                for (int k = 0; k < V; k++) fn(x[u].v[k]);
        }
        for (; i < whole; i += 32) {
            const Vec x = reinterpret_cast<const Vec *>(row)[i];
#pragma unroll
            for (int k = 0; k < V; k++) fn(x.v[k]);
        }
        for (i = whole * V + lane; i < G.nx; i += 32) fn(row[i]);
    }
}

// The maximum is exact in the state's own precision, and a NaN, once seen, is kept.
template <typename T>
__global__ void __launch_bounds__(256) hmax_kernel(Geom G, const T *h, Ctrl *ctrl)
{
    __shared__ double red[32];
    T m = T(0);
    for_depths(G, h, [&](T v) { m = (v > m || v != v) ? v : m; });
    const double bm = block_reduce<true>((double)m, red);
    if (threadIdx.x == 0) atomic_max_nonneg(&ctrl->hmax_bits, bm);
}

// Sum of a thread's share of the depths: FP64 state in double; FP32 state as
// an unevaluated float pair (s, c) by Knuth's branch-free two-sum, each
// addition's rounding error carried in c, so the pair holds the exact sum to
// about n u^2 of the summands (n per thread, u = 2^-24) and the FP64 pipe is
// left out of the per-element work.
template <typename T>
struct ThreadSum;

template <>
struct ThreadSum<double> {
    double s = 0.0;
    __device__ void add(double x) { s += x; }
    __device__ double value() const { return s; }
};

template <>
struct ThreadSum<float> {
    float s = 0.0f, c = 0.0f;
    __device__ void add(float x)
    {
        const float t = __fadd_rn(s, x);
        const float bp = __fsub_rn(t, s);
        const float e = __fadd_rn(__fsub_rn(s, __fsub_rn(t, bp)), __fsub_rn(x, bp));
        c = __fadd_rn(c, e);
        s = t;
    }
    __device__ double value() const { return (double)s + (double)c; }
};

// Pass 1: a fixed share of the rows per block (fixed order for a fixed launch shape).
template <typename T>
__global__ void __launch_bounds__(256) volume_partial_kernel(Geom G, const T *h, double *partials)
{
    __shared__ double red[32];
    ThreadSum<T> acc;
    for_depths(G, h, [&](T v) { acc.add(v); });
    const double s = block_reduce<false>(acc.value(), red);
    if (threadIdx.x == 0) partials[blockIdx.x] = s;
}

__global__ void volume_final_kernel(const double *partials, int np, double area, double *out)
{
    __shared__ double red[32];
    double s = 0.0;
    for (int k = threadIdx.x; k < np; k += blockDim.x) s += partials[k];
    s = block_reduce<false>(s, red);
    if (threadIdx.x == 0) *out = s * area;
}

template <typename T>
__global__ void gauges_kernel(Geom G, const T *h, const int64_t *cells, int ng, double *out)
{
    int k = blockIdx.x * blockDim.x + threadIdx.x;
    if (k >= ng) return;
    int64_t c = cells[k];
    out[k] = (double)h[(c / G.nx) * G.pitch + (c % G.nx)];
}

__global__ void __launch_bounds__(128)
    gauge_rows_kernel(Geom G, const float *rows, int n_rows, const int *row, const int64_t *cells, int ng, int64_t n, double *out)
{
    pdl_wait();
    pdl_launch();
    for (int64_t x = blockIdx.x * 128LL + threadIdx.x; x < n; x += gridDim.x * 128LL) {
        const int64_t s = x / ng, c = cells[x - s * ng];
        const int j = (int)(c / G.nx);
        out[x] = (double)rows[((size_t)s * n_rows + row[j]) * G.pitch + (c - (int64_t)j * G.nx)];
    }
}

}  // namespace

// Parts of a decomposed grid: the largest of their running depth maxima
// (bits of non-negative doubles, or a NaN's larger bits) into every part, so
// that each part's epoch start takes the whole grid's h_max.
__global__ void hmax_allreduce_kernel(Ctrl *const *ctrls, int n)
{
    if (threadIdx.x != 0 || blockIdx.x != 0) return;
    unsigned long long m = 0ull;
    for (int k = 0; k < n; k++) m = ctrls[k]->hmax_bits > m ? ctrls[k]->hmax_bits : m;
    for (int k = 0; k < n; k++) ctrls[k]->hmax_bits = m;
}

cudaError_t launch_hmax_allreduce(Ctrl *const *ctrls, int n, cudaStream_t st)
{
    hmax_allreduce_kernel<<<1, 32, 0, st>>>(ctrls, n);
    return cudaGetLastError();
}

static cudaError_t launch_epoch_begin(const Geom &g, Ctrl *ctrl, double *t_list, int E, const double *fixed_dt,
                                      cudaStream_t st)
{
    epoch_begin_kernel<<<1, 32, 0, st>>>(g, ctrl, t_list, E, fixed_dt);
    return cudaGetLastError();
}

template <typename T>
cudaError_t launch_epoch_batched(const EpochArgs<T> *tab, int n, const int2 *tasks, int n_tasks, int E, bool all_inflow,
                                 cudaStream_t st)
{
    if (all_inflow) {
        inflow_batched_kernel<T, true><<<dim3(E, n_tasks), kInflowThreads, 0, st>>>(tab, tasks);
        return cudaGetLastError();
    }
    epoch_begin_batched_kernel<T><<<(n + 127) / 128, 128, 0, st>>>(tab, n, E);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess || n_tasks == 0) return e;
    inflow_batched_kernel<T, false><<<dim3(E, n_tasks), kInflowThreads, 0, st>>>(tab, tasks);
    return cudaGetLastError();
}

template cudaError_t launch_epoch_batched<float>(const EpochArgs<float> *, int, const int2 *, int, int, bool,
                                                 cudaStream_t);

template <typename T>
cudaError_t launch_inflow(const EpochArgs<T> &A, int E, bool begin, const double *fixed_dt, cudaStream_t st)
{
    if (A.nsec == 0) return begin ? launch_epoch_begin(A.geo, A.ctrl, A.t_list, E, fixed_dt, st) : cudaSuccess;
    const dim3 grid(E, A.nsec);
    return launch_pdl(begin ? inflow_kernel<T, true> : inflow_kernel<T, false>, grid, kInflowThreads, st, A.geo, A.ctrl,
                      fixed_dt, A.secs, A.nsec, A.cells, A.tab_t, A.tab_q, A.z, A.n, A.t_list, E, A.inflow_q, A.n_slots,
                      A.inflow_Q, A.inflow_W);
}

template <typename T>
cudaError_t launch_hmax(const Geom &g, const T *h, Ctrl *ctrl, cudaStream_t st)
{
    const int rows = (g.ny + 7) / 8, blocks = rows < 152 * 8 ? rows : 152 * 8;   // a row per warp
    hmax_kernel<T><<<blocks, 256, 0, st>>>(g, h, ctrl);
    return cudaGetLastError();
}

template <typename T>
cudaError_t launch_volume(const Geom &g, const T *h, double *partials, int n_partials, double *out,
                          cudaStream_t st)
{
    const int rows = (g.ny + 7) / 8, blocks = rows < 1 ? 1 : rows < n_partials ? rows : n_partials;   // a row per warp
    volume_partial_kernel<T><<<blocks, 256, 0, st>>>(g, h, partials);
    volume_final_kernel<<<1, 256, 0, st>>>(partials, blocks, g.dx * g.dx, out);
    return cudaGetLastError();
}

// Non-finite values among rows x cols elements of a pitched array: OR of the
// test into *flag (rows grid-strided over blocks, columns over threads).
template <typename T>
__global__ void nonfinite_kernel(const T *a, int rows, int cols, int pitch, int *flag)
{
    int bad = 0;
    for (int r = blockIdx.x; r < rows; r += gridDim.x) {
        const T *row = a + (size_t)r * pitch;
        for (int c = threadIdx.x; c < cols; c += blockDim.x) bad |= !isfinite(row[c]);
    }
    if (__syncthreads_or(bad) && threadIdx.x == 0) atomicOr(flag, 1);
}

template <typename T>
cudaError_t launch_nonfinite(const T *a, int rows, int cols, int pitch, int *flag, cudaStream_t st)
{
    const int blocks = rows < 152 * 8 ? rows : 152 * 8;
    nonfinite_kernel<T><<<blocks, 256, 0, st>>>(a, rows, cols, pitch, flag);
    return cudaGetLastError();
}

// Poison of the pitch padding: quiet NaNs with a fixed payload, compared by bits.
template <typename U>
__global__ void padding_kernel(U *a, int rows, int cols, int pitch, U poison, int fill, unsigned long long *count)
{
    const int w = pitch - cols;
    unsigned long long bad = 0;
    for (long long k = blockIdx.x * (long long)blockDim.x + threadIdx.x; k < (long long)rows * w;
         k += (long long)gridDim.x * blockDim.x) {
        U *p = a + (size_t)(k / w) * pitch + cols + (k % w);
        if (fill) *p = poison;
        else bad += *p != poison;
    }
    if (!fill && bad) atomicAdd(count, bad);
}

cudaError_t launch_padding(void *a, size_t esz, int rows, int cols, int pitch, bool fill,
                           unsigned long long *count, cudaStream_t st)
{
    if (pitch <= cols || rows <= 0) return cudaSuccess;
    const long long n = (long long)rows * (pitch - cols);
    const int blocks = (int)(n < 152 * 8 * 256 ? (n + 255) / 256 : 152 * 8);
    if (esz == 4)
        padding_kernel<unsigned><<<blocks, 256, 0, st>>>((unsigned *)a, rows, cols, pitch, 0x7fc0deadu, fill ? 1 : 0,
                                                         count);
    else
        padding_kernel<unsigned long long><<<blocks, 256, 0, st>>>((unsigned long long *)a, rows, cols, pitch,
                                                                   0x7ff80000deadbeefull, fill ? 1 : 0, count);
    return cudaGetLastError();
}

template <typename T>
cudaError_t launch_gauges(const Geom &g, const T *h, const int64_t *cells, int G, double *out,
                          cudaStream_t st)
{
    if (G <= 0) return cudaSuccess;
    gauges_kernel<T><<<(G + 127) / 128, 128, 0, st>>>(g, h, cells, G, out);
    return cudaGetLastError();
}

cudaError_t launch_gauge_rows(const Geom &g, const float *rows, int n_rows, const int *row, const int64_t *cells, int G,
                              int n_steps, double *out, cudaStream_t st)
{
    const int64_t n = (int64_t)n_steps * G, blocks = (n + 127) / 128;
    if (n <= 0) return cudaSuccess;
    return launch_pdl(gauge_rows_kernel, (unsigned)(blocks < 152 * 16 ? blocks : 152 * 16), 128, st, g, rows, n_rows, row, cells, G, n,
                      out);
}

#define FLOOD_INST(T)                                                                                      \
    template cudaError_t launch_inflow<T>(const EpochArgs<T> &, int, bool, const double *, cudaStream_t);       \
    template cudaError_t launch_hmax<T>(const Geom &, const T *, Ctrl *, cudaStream_t);                     \
    template cudaError_t launch_volume<T>(const Geom &, const T *, double *, int, double *, cudaStream_t);   \
    template cudaError_t launch_gauges<T>(const Geom &, const T *, const int64_t *, int, double *, cudaStream_t); \
    template cudaError_t launch_nonfinite<T>(const T *, int, int, int, int *, cudaStream_t);
FLOOD_INST(float)
FLOOD_INST(double)
#undef FLOOD_INST

}  // namespace flood
