// step_reference.cu -- every operation IEEE-rounded in the order of the plain
// definition (Methods, Eq. 3-4, boundary faces by Eq. 5-6).  This is the FP64 path
// and the FP32 cross-check.
//
// A warp walks a chunk of rows of a strip of 31 columns, south to north, one column
// per lane: at row j it computes the row's south faces, finishes row j - 1 (Eq. 4) and
// computes the row's west faces; lane 31 adds the west face of the next strip's first
// column, which is the last cell's east face.  So each face is computed once (31/32 of
// the x-faces' lanes and rows/(rows + 1) of the y-faces are new), and both cells take
// the same bits, so the update conserves mass exactly like the face-by-face definition.
//
// FP64 is bound by its pipe: two operations a cycle and SM, about 55 per wet face
// (two divisions and a cube root; the division by dx takes three, Divisor).  A dry face takes its
// maxima and its test on the integer units, and a cell between four dry faces keeps its depth, so dry
// land costs four operations a cell.  A thread per cell computing its four faces itself took 274 us a step
// at 1001 x 777 (30 % wet; now 114, 130 with the ordinary division by dx), 36 at 128^2 (now 14.5).
#include "device_common.cuh"
#include "pdl.cuh"

namespace flood {

namespace {

constexpr int kCols = 31;

template <typename T>
__device__ __forceinline__ T boundary_face(const StepArgs<T> &a, int side, int k, T h_cell, T n_cell,
                                           double &vout)
{
    const Geom &G = a.geo;
    int off = side == 0 ? 0 : side == 1 ? G.ny : side == 2 ? 2 * G.ny : 2 * G.ny + G.nx;
    int type = a.bc.type[off + k];
    if (type == kBcWall) return T(0);
    T inward = T(inward_sign(side));
    if (type == kBcInflow) return inward * a.inflow_q[(size_t)a.s * a.n_slots + a.bc.slot[off + k]];
    T q = outflow_flux_ieee<T>(h_cell, T(a.bc.sqrtS[off + k]), n_cell, T(G.dx), T(G.h_dry), G.bc_form);
    if (type == kBcOutflow) vout += (double)q * G.dx;
    return -inward * q;
}

// Maximum and comparison of doubles on the integer units: 64-bit integers order like the doubles of their
// sign, and a dry face, whose flow depth and wet/dry test are all it has, would spend three quarters of its
// FP64 operations on them.  fmax's rule for NaN: the other operand.
__device__ __forceinline__ float max_of(float a, float b) { return fmaxf(a, b); }

__device__ __forceinline__ double max_of(double a, double b)
{
    const long long x = __double_as_longlong(a), y = __double_as_longlong(b);
    const bool both = (x & y) < 0;                     // both negative: the larger bits are the smaller number
    const bool first = both ? x < y : x > y;
    const long long big = first ? x : y, other = first ? y : x;
    const bool nan = (big & 0x7fffffffffffffffll) > 0x7ff0000000000000ll;
    // a NaN of either sign sorts above every number of its sign, or below them all
    return __longlong_as_double(nan ? other : big);
}

// hf > hd for hd > 0 (false for NaN).
__device__ __forceinline__ bool above(float hf, float hd) { return hf > hd; }

__device__ __forceinline__ bool above(double hf, double hd)
{
    const long long x = __double_as_longlong(hf);
    return x > __double_as_longlong(hd) && x <= 0x7ff0000000000000ll;
}

__device__ __forceinline__ bool all_zero(float a, float b, float c, float d)
{
    return a == 0.0f && b == 0.0f && c == 0.0f && d == 0.0f;
}

__device__ __forceinline__ bool all_zero(double a, double b, double c, double d)
{
    return ((__double_as_longlong(a) | __double_as_longlong(b) | __double_as_longlong(c) | __double_as_longlong(d)) << 1) == 0;
}

// Item (strip, chunk) = (block % n_strips, block / n_strips).
template <typename T>
__global__ void __launch_bounds__(32) step_reference_kernel(const __grid_constant__ StepArgs<T> a, const int n_strips, const int rows)
{
    using O = R<T>;
    pdl_wait();
    pdl_launch();
    const Geom &G = a.geo;
    const int nx = G.nx, ny = G.ny, lane = threadIdx.x;
    const int x0 = (int)(blockIdx.x % (unsigned)n_strips) * kCols, c = x0 + lane;
    const int y0 = (int)(blockIdx.x / (unsigned)n_strips) * rows, y1 = min(y0 + rows, ny);
    const size_t P = (size_t)G.pitch;
    const T dt = T(a.ctrl->dt), g = T(G.g), hd = T(G.h_dry);
    const Divisor<T> dx(T(G.dx));
    const bool wt = G.theta != 1.0;                   // theta-weighted numerator discharges
    const bool vec = G.friction != 0;                 // vector-norm |q| in the friction term
    const T th = T(G.theta), w = T(0.5 * (1.0 - G.theta));
    const bool cell = c < nx, own = cell && lane < kCols;   // lane 31's cell belongs to the next strip
    const T *qx = a.qx, *qy = a.qy;
    double vout = 0.0, vclip = 0.0, hmax = 0.0;
    T hp = T(0), zp = T(0), np_ = T(0), ep = T(0);    // row j - 1: depth, bed, n, water level,
    T xp = T(0), yp = T(0);                           // new west and south faces
    if (y0 > 0 && own) {
        const size_t r = (size_t)(y0 - 1) * P + c;
        hp = a.h[r];
        zp = a.z[r];
        np_ = a.n[r];
        ep = O::add(hp, zp);
    }
    for (int j = y0; j <= y1; j++) {
        const size_t r = (size_t)j * P + c;
        T hC = T(0), zC = T(0), nC = T(0);
        if (j < ny && cell) {
            hC = a.h[r];
            zC = a.z[r];
            nC = a.n[r];
        }
        const T eC = O::add(hC, zC);
        // ---- south faces of row j (interior y-faces j in 1..ny-1 have neighbours j-1 >= 0 and j+1 <= ny and
        // x-faces of columns c, c+1 <= nx in rows j-1, j)
        T ys = T(0);
        if (own) {
            if (j == 0) ys = boundary_face(a, 2, c, hC, nC, vout);
            else if (j == ny) ys = boundary_face(a, 3, c, hp, np_, vout);
            else {
                const T hf = O::sub(max_of(ep, eC), max_of(zp, zC));
                if (above(hf, hd))
                    ys = face_wet_ieee<T>(wt ? theta_q_ieee<T>(qy[r], qy[r - P], qy[r + P], th, w, true) : qy[r],
                                          vec ? q_norm_ieee<T>(qy[r], qx[r - P], qx[r - P + 1], qx[r], qx[r + 1], true)
                                              : R<T>::abs(qy[r]),
                                          ep, eC, hf, np_, nC, g, dt, dx);
            }
        }
        // ---- finish row j-1: Eq. 4 with the new fluxes, then the depth clip
        if (j > y0) {
            const T xe = __shfl_down_sync(0xffffffffu, xp, 1);
            if (own) {
                T hn = hp;                              // four dry faces: hp + dt 0 / dx
                if (!all_zero(xp, xe, yp, ys)) {
                    const T dv = O::add(O::sub(xp, xe), O::sub(yp, ys));
                    hn = O::add(hp, dx.under(O::mul(dt, dv)));
                }
                if (hn < T(0)) {
                    if (j - 1 >= G.led_j0 && j - 1 < G.led_j1) vclip += -(double)hn * G.dx * G.dx;
                    hn = T(0);
                }
                a.h_out[r - P] = hn;
                a.qy_out[r - P] = yp;
                if (j == ny) a.qy_out[r] = ys;
                if (a.want_hmax) hmax = nanmax(hmax, (double)hn);
            }
            if (own || c == nx) a.qx_out[r - P] = xp;
        }
        // ---- west faces of row j (interior x-faces c in 1..nx-1 have neighbours c-1 >= 0 and c+1 <= nx in the row
        // and y-faces of columns c-1, c in rows j, j+1 <= ny)
        if (j < y1) {
            T hL = __shfl_up_sync(0xffffffffu, hC, 1), zL = __shfl_up_sync(0xffffffffu, zC, 1),
              nL = __shfl_up_sync(0xffffffffu, nC, 1), eL = __shfl_up_sync(0xffffffffu, eC, 1);
            if (lane == 0 && c > 0) {
                hL = a.h[r - 1];
                zL = a.z[r - 1];
                nL = a.n[r - 1];
                eL = O::add(hL, zL);
            }
            xp = T(0);
            if (c == 0) xp = boundary_face(a, 0, j, hC, nC, vout);
            else if (c == nx) xp = boundary_face(a, 1, j, hL, nL, vout);
            else if (cell) {
                const T hf = O::sub(max_of(eL, eC), max_of(zL, zC));
                if (above(hf, hd))
                    xp = face_wet_ieee<T>(wt ? theta_q_ieee<T>(qx[r], qx[r - 1], qx[r + 1], th, w, true) : qx[r],
                                          vec ? q_norm_ieee<T>(qx[r], qy[r - 1], qy[r], qy[r + P - 1], qy[r + P], true)
                                              : R<T>::abs(qx[r]),
                                          eL, eC, hf, nL, nC, g, dt, dx);
            }
            hp = hC;
            zp = zC;
            np_ = nC;
            ep = eC;
            yp = ys;
        }
    }
    // ledger: outflow and clip volumes (an atomic for a warp that has any)
    if (__any_sync(0xffffffffu, vout != 0.0)) {
        vout = warp_sum(vout);
        if (lane == 0) atomicAdd(&a.ctrl->V_out, (double)dt * vout);
    }
    if (__any_sync(0xffffffffu, vclip != 0.0)) {
        vclip = warp_sum(vclip);
        if (lane == 0) atomicAdd(&a.ctrl->V_clip, vclip);
    }
    if (a.want_hmax) {
        hmax = warp_max(hmax);
        if (lane == 0) atomic_max_nonneg(&a.ctrl->hmax_bits, hmax);
    }
    if (blockIdx.x == 0 && lane == 0) {
        double vin = a.ctrl->V_in;
        for (int k = 0; k < a.n_inflow_sec; k++) {
            double Q = a.inflow_Q[(size_t)a.s * a.n_inflow_sec + k];
            if (Q > 0.0) vin += a.ctrl->dt * Q;
        }
        a.ctrl->V_in = vin;
        a.ctrl->t = a.t_list[a.s + 1];
    }
}

// Rows per item: an item of r rows computes 2 r + 1 rows of faces, but the FP64 pipes even out over many short items,
// whose wet ones cluster.  us a step at 1 / 2 / 3 rows, 30 % and 90 % wet: 17.7 / 26.0 / 34.6 and 19.5 / 26.1 / 34.6
// (128^2), 32 / 29 / 36 and 42 / 38 / 44 (256^2), 38 / 49 / 40 and 65 / 66 / 66 (360^2), 58 / 58 / 70 and 103 / 102 / 90 (512^2),
// 78 / 70 / 79 and 150 / 140 / 141 (640^2), 94 / 88 / 82 and 186 / 161 / 158 (720^2), 136 / 116 / 121 and 269 / 232 / 218
// (1001 x 777), 173 / 143 / 137 and 357 / 299 / 283 (1024^2), 228 / 184 / 175 and 475 / 395 / 371 (1200^2): one row up to where
// two draw level for good, three from where they lead at either wetness.
int reference_rows(int nx, int ny)
{
    const int64_t cells = (int64_t)nx * ny;
    return cells < (1 << 18) ? 1 : cells < (1 << 20) ? 2 : 3;
}

}  // namespace

template <typename T>
cudaError_t launch_step_reference(const StepArgs<T> &a, cudaStream_t st)
{
    const int n_strips = (a.geo.nx + kCols - 1) / kCols;
    const int rows = reference_rows(a.geo.nx, a.geo.ny);
    const int64_t items = (int64_t)n_strips * ((a.geo.ny + rows - 1) / rows);
    const cudaError_t e = launch_pdl(step_reference_kernel<T>, (unsigned)items, 32, st, a, n_strips, rows);
    if (e != cudaSuccess || !a.gauge_out) return e;
    return launch_gauges<T>(a.geo, a.h_out, a.gauge_cells, a.n_gauges, a.gauge_out, st);
}

template cudaError_t launch_step_reference<float>(const StepArgs<float> &, cudaStream_t);
template cudaError_t launch_step_reference<double>(const StepArgs<double> &, cudaStream_t);

}  // namespace flood
