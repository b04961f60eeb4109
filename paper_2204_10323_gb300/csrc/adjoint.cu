// adjoint.cu -- reverse of one time step (not in the paper; its calibration
// use is named as future work).  Given the forward state x_k and the adjoint
// lambda_{k+1} of the state after the step, produce lambda_k and accumulate
// dL/dn.  The forward step is h' = max(h + dt/dx div q'(x_k, n), 0) with q'
// from Eq. 3 on interior faces and Eq. 5-6 on boundary faces, so
//
//   lambda_hu(c) = lambda_h'(c) * [h'_unclipped(c) >= 0]
//   mu_f         = lambda_q'(f) + dt/dx (lambda_hu(R) - lambda_hu(L))     (face f between L and R)
//   lambda_h(c)  = lambda_hu(c) + sum_f mu_f dq'_f/dh_c
//   lambda_q(f)  = mu_f dq'_f/dq_f                                          (interior faces)
//   dL/dn(c)    += sum_f mu_f dq'_f/dn_c
//
// Branch conventions: max(eta_L, eta_R) sends its derivative to L on ties;
// d|q|/dq = 0 at q = 0; the dry-face test, the outflow dry test and the clip
// are held as masks; the Eq. 6 level is differentiated exactly through the
// implicit function theorem.  Each cell gathers the contributions of its
// four faces (both cells of a face evaluate its derivatives), so no atomics
// are needed and the result is deterministic.
//
// The clip mask is recomputed with the forward kernels' own arithmetic (IEEE
// order for FP64, the fast FP32 face for FP32), so the clip and wet/dry
// decisions are exactly the forward's.
#include <algorithm>
#include <cstddef>
#include <type_traits>

#include "fast_face.cuh"
#include "step_tiled.cuh"

namespace flood {

namespace {

constexpr int BX = 32;

// ---------------------------------------------------------------- forward faces per precision
template <typename T> struct Fwd;

template <> struct Fwd<double> {
    double g, dt, dx, hd;
    Divisor<double> over_dx;
    __device__ Fwd(const Geom &G, double dt_) : g(G.g), dt(dt_), dx(G.dx), hd(G.h_dry), over_dx(G.dx) {}
    __device__ double face(double q, double hL, double zL, double nL, double hR, double zR, double nR) const
    {
        return face_update_ieee<double>(q, fabs(q), hL, zL, nL, hR, zR, nR, g, dt, over_dx, hd);
    }
    __device__ double hf(double hL, double zL, double hR, double zR) const
    {
        using O = R<double>;
        return O::sub(O::max(O::add(hL, zL), O::add(hR, zR)), O::max(zL, zR));
    }
    __device__ double outflow(double h, double sqrtS, double n, int form) const
    {
        return outflow_flux_ieee<double>(h, sqrtS, n, dx, hd, form);
    }
    __device__ double update(double h, double qW, double qE, double qS, double qN) const
    {
        using O = R<double>;
        double dv = O::add(O::sub(qW, qE), O::sub(qS, qN));
        return O::add(h, over_dx.under(O::mul(dt, dv)));
    }
    __device__ static double rcp_(double x) { return 1.0 / x; }
    __device__ static double pow_m73_(double x) { const double m = ::rcbrt(x), r = 1.0 / x; return m * r * r; }
};

template <> struct Fwd<float> {
    FastConst K;
    float dx, hd;
    __device__ Fwd(const Geom &G, double dt_)
    {
        const float dt = (float)dt_;
        dx = (float)G.dx;
        K.gdt = (float)G.g * dt;
        K.a1 = K.gdt / dx;
        K.gdt4 = 0.25f * K.gdt;
        K.h_dry = (float)G.h_dry;
        K.dtdx = dt / dx;
        hd = K.h_dry;
    }
    __device__ float face(float q, float hL, float zL, float nL, float hR, float zR, float nR) const
    {
        return face_fast(q, hL + zL, hR + zR, fmaxf(zL, zR), nL + nR, K);
    }
    __device__ float hf(float hL, float zL, float hR, float zR) const
    {
        return __fsub_rn(fmaxf(hL + zL, hR + zR), fmaxf(zL, zR));
    }
    __device__ float outflow(float h, float sqrtS, float n, int form) const
    {
        return outflow_fast(h, sqrtS, n, dx, hd, form);
    }
    __device__ float update(float h, float qW, float qE, float qS, float qN) const
    {
        float dv = __fadd_rn(__fsub_rn(qW, qE), __fsub_rn(qS, qN));
        return __fmaf_rn(K.dtdx, dv, h);
    }
    __device__ static float rcp_(float x) { return rcp_fast(x); }
    __device__ static float pow_m73_(float x) { return pow_m73(x); }
};

// Partial derivatives of one wet face's Eq. 3 value.
template <typename T> struct FaceLin {
    T dq, dhL, dhR, dn;     // dn = dq'/dn_L = dq'/dn_R
};

template <typename T>
__device__ __forceinline__ FaceLin<T> face_lin(T q, T hL, T zL, T nL, T hR, T zR, T nR, T hf, T g, T dt, T dx)
{
    FaceLin<T> r;
    const T etaL = hL + zL, etaR = hR + zR;
    const T nf = T(0.5) * (nL + nR);
    const T gdt = g * dt, a1 = gdt / dx;
    const T inv_hf = Fwd<T>::rcp_(hf);
    const T hf_m73 = Fwd<T>::pow_m73_(hf);
    const T c0 = gdt * nf * nf * hf_m73;     // friction per |q|
    const T fric = c0 * (q < T(0) ? -q : q);
    const T inv_den = Fwd<T>::rcp_(T(1) + fric);
    const T slope = etaR - etaL;
    const T F = (q - a1 * hf * slope) * inv_den;
    const T sg = q > T(0) ? T(1) : (q < T(0) ? T(-1) : T(0));
    r.dq = (T(1) - F * c0 * sg) * inv_den;
    const T dF_dhf = (-a1 * slope + F * (T(7) / T(3)) * fric * inv_hf) * inv_den;
    const T d_expl = a1 * hf * inv_den;
    const bool left = etaL >= etaR;
    r.dhL = d_expl + (left ? dF_dhf : T(0));
    r.dhR = -d_expl + (left ? T(0) : dF_dhf);
    r.dn = -F * fric * inv_den * Fwd<T>::rcp_(nf);
    return r;
}

template <typename T>
__device__ __forceinline__ int bc_off(const Geom &G, int side)
{
    return side == 0 ? 0 : side == 1 ? G.ny : side == 2 ? 2 * G.ny : 2 * G.ny + G.nx;
}

// Forward boundary face value (same rules as the forward kernels).
template <typename T>
__device__ __forceinline__ T bface(const StepArgs<T> &a, const Fwd<T> &F, int side, int k, T h, T n)
{
    const Geom &G = a.geo;
    const int off = bc_off<T>(G, side);
    const int type = a.bc.type[off + k];
    if (type == kBcWall) return T(0);
    const T inward = T(inward_sign(side));
    if (type == kBcInflow) return inward * a.inflow_q[(size_t)a.s * a.n_slots + a.bc.slot[off + k]];
    return -inward * F.outflow(h, T(a.bc.sqrtS[off + k]), n, G.bc_form);
}

// Adjoint of an outflow boundary face: contributions to lambda_h(c) and dL/dn(c).
template <typename T>
__device__ __forceinline__ void outflow_adj(const StepArgs<T> &a, const Fwd<T> &F, int side, int k, T h, T n,
                                            T mu, T &lh, T &gn)
{
    const Geom &G = a.geo;
    const int off = bc_off<T>(G, side);
    if (a.bc.type[off + k] != kBcOutflow) return;
    const T q = F.outflow(h, T(a.bc.sqrtS[off + k]), n, G.bc_form);
    if (!(q > T(0))) return;                    // dry boundary cell: held at zero
    const T nu = -T(inward_sign(side)) * mu;   // adjoint of the outflow magnitude
    const T pe = G.bc_form == 0 ? T(5.0 / 3.0) : T(2.0 / 3.0);
    lh += nu * pe * q / h;
    gn += -nu * q / n;
}

// One launch per reverse step, face-centric within a BX x 8 tile (256
// threads: 32 registers and 19 KB of shared memory in FP32 let eight blocks
// share an SM, so one block's barriers and loads overlap the others' work;
// 32 x 16 and 32 x 4 tiles measured 12 % and 15 % slower at 1024^2):
//  0. the tile's cells with a two-cell halo (h, z, n) and the faces around it
//     (old q) are staged in shared memory;
//  A. every face around the tile and its one-cell halo gets its new value q'
//     (the forward arithmetic);
//  B. the tile and halo cells get the adjoint of their unclipped depth
//     (lambda_h' plus the gauge seeds, zero where the depth was clipped);
//  C. every face touching a tile cell gets mu and its derivatives once,
//     leaving its contributions to the two cells and the adjoint of its old q;
//  D. every tile cell gathers the contributions of its four faces.
template <typename T> struct TileRows { static constexpr int v = 8; };
constexpr int kTileGauges = 32;

template <typename T>
__global__ void __launch_bounds__(BX * TileRows<T>::v) adj_step_kernel(const AdjArgs<T> A, const int nbx)
{
    constexpr int BYT = TileRows<T>::v;
    constexpr int NT = BX * BYT;
    __shared__ T sh[BYT + 4][BX + 4], sz[BYT + 4][BX + 4], sn[BYT + 4][BX + 4];   // cells I0-2.., J0-2..
    __shared__ T sqx[BYT + 2][BX + 3], sX[BYT + 2][BX + 3];   // x-faces: columns I0-1 .., rows J0-1 ..
    __shared__ T sqy[BYT + 3][BX + 2], sY[BYT + 3][BX + 2];   // y-faces: rows J0-1 .., columns I0-1 ..
    __shared__ T sL[BYT + 2][BX + 2];                          // cells I0-1 .., J0-1 ..
    __shared__ T cXl[BYT][BX + 1], cXr[BYT][BX + 1], cXn[BYT][BX + 1];
    __shared__ T cYl[BYT + 1][BX], cYr[BYT + 1][BX], cYn[BYT + 1][BX];
    __shared__ int s_ng, s_gk[kTileGauges];                     // gauges inside the tile and its halo
    const StepArgs<T> &a = A.fwd;
    const Geom &G = a.geo;
    const int nx = G.nx, ny = G.ny;
    const size_t P = (size_t)G.pitch;
    const double dtd = a.ctrl->dt;
    const Fwd<T> F(G, dtd);
    const T dt = T(dtd), dx = T(G.dx), g = T(G.g), hd = T(G.h_dry), dtdx = dt / dx;
    const int tid = threadIdx.y * BX + threadIdx.x;
    // one-dimensional grid (grids taller than 65535 tiles): tile (bx, by) of nbx columns of tiles
    const int I0 = (int)(blockIdx.x % (unsigned)nbx) * BX, J0 = (int)(blockIdx.x / (unsigned)nbx) * BYT;

    // 0. stage cells and old face fluxes (zeros outside the domain)
    for (int t = tid; t < (BYT + 4) * (BX + 4); t += NT) {
        const int lj = t / (BX + 4), li = t % (BX + 4);
        const int j = J0 - 2 + lj, i = I0 - 2 + li;
        T hv = T(0), zv = T(0), nv = T(0);
        if (i >= 0 && i < nx && j >= 0 && j < ny) {
            const size_t c = (size_t)j * P + i;
            hv = a.h[c];
            zv = a.z[c];
            nv = a.n[c];
        }
        sh[lj][li] = hv;
        sz[lj][li] = zv;
        sn[lj][li] = nv;
    }
    for (int t = tid; t < (BYT + 2) * (BX + 3); t += NT) {
        const int lj = t / (BX + 3), li = t % (BX + 3);
        const int j = J0 - 1 + lj, fi = I0 - 1 + li;
        sqx[lj][li] = (j >= 0 && j < ny && fi >= 0 && fi <= nx) ? a.qx[(size_t)j * P + fi] : T(0);
    }
    for (int t = tid; t < (BYT + 3) * (BX + 2); t += NT) {
        const int lj = t / (BX + 2), li = t % (BX + 2);
        const int fj = J0 - 1 + lj, i = I0 - 1 + li;
        sqy[lj][li] = (i >= 0 && i < nx && fj >= 0 && fj <= ny) ? a.qy[(size_t)fj * P + i] : T(0);
    }
    __syncthreads();
    // A. new face values.  x-face (lj, li) lies between cells (lj+1, li) and (lj+1, li+1) of the staging.
    for (int t = tid; t < (BYT + 2) * (BX + 3); t += NT) {
        const int lj = t / (BX + 3), li = t % (BX + 3);
        const int j = J0 - 1 + lj, fi = I0 - 1 + li;
        T v = T(0);
        if (j >= 0 && j < ny && fi >= 0 && fi <= nx) {
            const int sj = lj + 1, sl = li, sr = li + 1;
            if (fi == 0) v = bface(a, F, 0, j, sh[sj][sr], sn[sj][sr]);
            else if (fi == nx) v = bface(a, F, 1, j, sh[sj][sl], sn[sj][sl]);
            else v = F.face(sqx[lj][li], sh[sj][sl], sz[sj][sl], sn[sj][sl], sh[sj][sr], sz[sj][sr], sn[sj][sr]);
        }
        sX[lj][li] = v;
    }
    // y-face (lj, li) lies between cells (lj, li+1) and (lj+1, li+1) of the staging.
    for (int t = tid; t < (BYT + 3) * (BX + 2); t += NT) {
        const int lj = t / (BX + 2), li = t % (BX + 2);
        const int fj = J0 - 1 + lj, i = I0 - 1 + li;
        T v = T(0);
        if (i >= 0 && i < nx && fj >= 0 && fj <= ny) {
            const int sc = li + 1, sb = lj, st = lj + 1;
            if (fj == 0) v = bface(a, F, 2, i, sh[st][sc], sn[st][sc]);
            else if (fj == ny) v = bface(a, F, 3, i, sh[sb][sc], sn[sb][sc]);
            else v = F.face(sqy[lj][li], sh[sb][sc], sz[sb][sc], sn[sb][sc], sh[st][sc], sz[st][sc], sn[st][sc]);
        }
        sY[lj][li] = v;
    }
    __syncthreads();
    // B. adjoint of the unclipped depth (gauge seeds included).  The gauges inside
    // the tile and its halo are listed first (flags in gauge order), so that a
    // cell scans only those; a tile holding more than kTileGauges scans them all.
    if (tid == 0) s_ng = 0;
    __syncthreads();
    for (int gk = tid; gk < A.n_gauges; gk += NT) {
        const int64_t flat = A.gauge_cells[gk];
        const int gj = (int)(flat / nx), gi = (int)(flat - (int64_t)gj * nx);
        if (gj >= J0 - 1 && gj <= J0 + BYT && gi >= I0 - 1 && gi <= I0 + BX) {
            const int slot = atomicAdd(&s_ng, 1);
            if (slot < kTileGauges) s_gk[slot] = gk;
        }
    }
    __syncthreads();
    if (tid == 0 && s_ng > 1 && s_ng <= kTileGauges) {   // restore gauge order: repeated gauges add up in order
        for (int x = 1; x < s_ng; x++)
            for (int y = x; y > 0 && s_gk[y - 1] > s_gk[y]; y--) {
                const int tmp = s_gk[y];
                s_gk[y] = s_gk[y - 1];
                s_gk[y - 1] = tmp;
            }
    }
    __syncthreads();
    const int ng_tile = s_ng;
    for (int t = tid; t < (BYT + 2) * (BX + 2); t += NT) {
        const int lj = t / (BX + 2), li = t % (BX + 2);
        const int j = J0 - 1 + lj, i = I0 - 1 + li;
        T v = T(0);
        if (i >= 0 && i < nx && j >= 0 && j < ny) {
            const T hu = F.update(sh[lj + 1][li + 1], sX[lj][li], sX[lj][li + 1], sY[lj][li], sY[lj + 1][li]);
            if (!(hu < T(0))) {
                v = A.lh[(size_t)j * P + i];
                if (ng_tile > 0) {
                    const int64_t flat = (int64_t)j * nx + i;
                    if (ng_tile <= kTileGauges) {
                        for (int x = 0; x < ng_tile; x++)
                            if (A.gauge_cells[s_gk[x]] == flat) v = v + T(A.seed[s_gk[x]]);
                    } else {
                        for (int gk = 0; gk < A.n_gauges; gk++)
                            if (A.gauge_cells[gk] == flat) v = v + T(A.seed[gk]);
                    }
                }
            }
        }
        sL[lj][li] = v;
    }
    __syncthreads();
    // C. each face touching the tile once.  x-face column li = fi - I0, row lj = j - J0.
    for (int t = tid; t < BYT * (BX + 1); t += NT) {
        const int lj = t / (BX + 1), li = t % (BX + 1);
        const int j = J0 + lj, fi = I0 + li;
        T cl = T(0), cr = T(0), cn = T(0);
        if (j < ny && fi <= nx) {
            const size_t r = (size_t)j * P;
            const T lR = sL[lj + 1][li + 1], lL = sL[lj + 1][li];
            const int sj = lj + 2, sl = li + 1, sr = li + 2;     // staging coordinates of L and R
            if (fi == 0) {
                const T mu = A.lqx[r] + dtdx * lR;
                outflow_adj(a, F, 0, j, sh[sj][sr], sn[sj][sr], mu, cr, cn);
                A.lqx_out[r] = T(0);
            } else if (fi == nx) {
                const T mu = A.lqx[r + nx] - dtdx * lL;
                outflow_adj(a, F, 1, j, sh[sj][sl], sn[sj][sl], mu, cl, cn);
                A.lqx_out[r + nx] = T(0);
            } else {
                const T mu = A.lqx[r + fi] + dtdx * (lR - lL);
                const T hL = sh[sj][sl], zL = sz[sj][sl], nL = sn[sj][sl];
                const T hR = sh[sj][sr], zR = sz[sj][sr], nR = sn[sj][sr];
                const T hf = F.hf(hL, zL, hR, zR);
                T lq = T(0);
                if (hf > hd && mu != T(0)) {
                    FaceLin<T> d = face_lin<T>(sqx[lj + 1][li + 1], hL, zL, nL, hR, zR, nR, hf, g, dt, dx);
                    cl = mu * d.dhL;
                    cr = mu * d.dhR;
                    cn = mu * d.dn;
                    lq = mu * d.dq;
                }
                if (li < BX) A.lqx_out[r + fi] = lq;        // the tile owns the west faces of its cells
            }
        }
        cXl[lj][li] = cl;
        cXr[lj][li] = cr;
        cXn[lj][li] = cn;
    }
    // y-face row lj = fj - J0, column li = i - I0.
    for (int t = tid; t < (BYT + 1) * BX; t += NT) {
        const int lj = t / BX, li = t % BX;
        const int fj = J0 + lj, i = I0 + li;
        T cl = T(0), cr = T(0), cn = T(0);
        if (i < nx && fj <= ny) {
            const T lR = sL[lj + 1][li + 1], lL = sL[lj][li + 1];
            const int sc = li + 2, sb = lj + 1, st = lj + 2;     // staging coordinates of L (below) and R
            if (fj == 0) {
                const T mu = A.lqy[i] + dtdx * lR;
                outflow_adj(a, F, 2, i, sh[st][sc], sn[st][sc], mu, cr, cn);
                A.lqy_out[i] = T(0);
            } else if (fj == ny) {
                const size_t c = (size_t)(ny - 1) * P + i;
                const T mu = A.lqy[c + P] - dtdx * lL;
                outflow_adj(a, F, 3, i, sh[sb][sc], sn[sb][sc], mu, cl, cn);
                A.lqy_out[c + P] = T(0);
            } else {
                const size_t c = (size_t)fj * P + i;
                const T mu = A.lqy[c] + dtdx * (lR - lL);
                const T hL = sh[sb][sc], zL = sz[sb][sc], nL = sn[sb][sc];
                const T hR = sh[st][sc], zR = sz[st][sc], nR = sn[st][sc];
                const T hf = F.hf(hL, zL, hR, zR);
                T lq = T(0);
                if (hf > hd && mu != T(0)) {
                    FaceLin<T> d = face_lin<T>(sqy[lj + 1][li + 1], hL, zL, nL, hR, zR, nR, hf, g, dt, dx);
                    cl = mu * d.dhL;
                    cr = mu * d.dhR;
                    cn = mu * d.dn;
                    lq = mu * d.dq;
                }
                if (lj < BYT) A.lqy_out[c] = lq;            // the tile owns the south faces of its cells
            }
        }
        cYl[lj][li] = cl;
        cYr[lj][li] = cr;
        cYn[lj][li] = cn;
    }
    __syncthreads();
    // D. gather per tile cell
    const int tx = threadIdx.x, ty = threadIdx.y;
    const int i = I0 + tx, j = J0 + ty;
    if (i >= nx || j >= ny) return;
    const size_t c = (size_t)j * P + i;
    const T lu = sL[ty + 1][tx + 1];
    const T lh = lu + cXr[ty][tx] + cXl[ty][tx + 1] + cYr[ty][tx] + cYl[ty + 1][tx];
    // this step's dL/dn of the cell in the working precision, then one add into the
    // double accumulator over the sweep
    const T gs = (cXn[ty][tx] + cXn[ty][tx + 1]) + (cYn[ty][tx] + cYn[ty + 1][tx]);
    A.lh_out[c] = lh;
    A.gn[c] += (double)gs;
    if (i == 0 || j == 0 || i == nx - 1 || j == ny - 1) A.lhu[c] = lu;   // read by the inflow pass
}

// Pass 3: the inflow faces of each section depend on every section cell's n
// through the Eq. 6 level W: with w_c the cell discharge (sum_c w_c = Q),
// pe its depth exponent and hh_c = W - z_c,
//   dw_c/dn_j = -delta_cj w_c/n_c + (pe w_c/hh_c) dW/dn_j,
//   dW/dn_j   = (w_j/n_j) / sum_c (pe w_c/hh_c),
// so dL/dn_j += (w_j/n_j) (sum_c nu_c pe w_c/hh_c / sum_c pe w_c/hh_c - nu_j).

// Section k of pass 3 on the calling block (FP64 and the scheme options): reads lhu from the
// finished tiles and adds into gn.
template <typename T>
__device__ void inflow_adjoint(const AdjArgs<T> &A, const int k, double *red)
{
    const StepArgs<T> &a = A.fwd;
    const Geom &G = a.geo;
    const InflowSec S = A.secs[k];
    const double Q = a.inflow_Q[(size_t)a.s * a.n_inflow_sec + k];
    if (!(Q > 0.0) || S.ncell == 0) return;
    const double W = A.inflow_W[(size_t)a.s * a.n_inflow_sec + k];
    const double dx = G.dx, dtdx = a.ctrl->dt / G.dx;
    const double pe = G.bc_form == 0 ? 5.0 / 3.0 : 2.0 / 3.0;
    const double inward = (double)inward_sign(S.side);
    const size_t P = (size_t)G.pitch;
    const int tid = threadIdx.x + blockDim.x * threadIdx.y, nt = blockDim.x * blockDim.y;
    auto lhu_of = [&](int64_t idx) -> double { return (double)A.lhu[idx]; };
    auto lq_of = [&](int64_t idx) -> double {
        switch (S.side) {
        case 0: return (double)A.lqx[idx];
        case 1: return (double)A.lqx[idx + 1];
        case 2: return (double)A.lqy[idx];
        default: return (double)A.lqy[idx + P];
        }
    };
    double D = 0.0, Nn = 0.0, nu0 = 0.0;             // nu0: this thread's first cell (reused below)
    for (int c = tid; c < S.ncell; c += nt) {
        const int64_t idx = A.sec_cells[S.cell0 + c];
        const double hh = W - (double)a.z[idx];
        if (!(hh > 0.0)) continue;
        const double w = (double)a.inflow_q[(size_t)a.s * a.n_slots + S.slot0 + c] * dx;
        const double mu = lq_of(idx) + inward * dtdx * lhu_of(idx);
        const double nu = inward * mu / dx;
        if (c == tid) nu0 = nu;
        D += pe * w / hh;
        Nn += nu * pe * w / hh;
    }
    D = block_reduce<false>(D, red);
    __syncthreads();
    if (tid == 0) red[31] = D;
    __syncthreads();
    D = red[31];
    __syncthreads();
    Nn = block_reduce<false>(Nn, red);
    __syncthreads();
    if (tid == 0) red[30] = Nn;
    __syncthreads();
    Nn = red[30];
    if (!(D > 0.0)) return;
    for (int c = tid; c < S.ncell; c += nt) {
        const int64_t idx = A.sec_cells[S.cell0 + c];
        const double hh = W - (double)a.z[idx];
        if (!(hh > 0.0)) continue;
        const double w = (double)a.inflow_q[(size_t)a.s * a.n_slots + S.slot0 + c] * dx;
        const double nu = c == tid ? nu0 : inward * (lq_of(idx) + inward * dtdx * lhu_of(idx)) / dx;
        A.gn_in[S.slot0 + c] += (w / (double)a.n[idx]) * (Nn / D - nu);   // (sections may share a corner cell)
    }
}

template <typename T>
__global__ void adj_inflow_kernel(const AdjArgs<T> A)
{
    __shared__ double red[32];
    inflow_adjoint<T>(A, blockIdx.x, red);
}

// ---------------------------------------------------------------- FP32, Eq. 3 as printed
// The FP32 reverse step: one warp walks the rows of a strip of 60 output columns (64 staged, a
// pair per lane) south to north, as the temporal-blocking kernel does, in one pass.  At tick j:
//  A. row j's new faces (the forward arithmetic) and, from the same intermediates, each face's
//     derivatives with respect to its old discharge, its two depths and n; kept one tick;
//  B. the adjoint lu of row j-1's unclipped depth: its update needs the south faces of row j;
//  C. the x-faces of row j-1 and the y-faces between rows j-2 and j-1: mu, and its products with
//     the kept derivatives;
//  D. row j-2 is complete: its lambda_h and dL/dn.
// A border face keeps the derivatives of Eq. 5 in the same places (its outer cell has lu = 0), so
// that C and D know no borders; an inflow face leaves lu and lambda_q for pass 3.  Rows arrive by
// asynchronous copies, every lane's shared memory is its own: no barrier, no index arithmetic per
// element.
//
// A lone warp's chain bounds it (powers, reciprocals, shuffles, FP64 adds in series: six cycles an
// instruction), so a strip takes two columns per lane where the forward kernel takes four: half the instructions
// a tick and twice the warps.  A sweep of 64 steps with its states kept, two / four columns: 2.07 / 2.23 ms
// (1024^2), 1.27 / 1.59 (512^2), 1.08 / 1.56 (256^2), 5.74 / 6.08 (2048^2).  A step of 1024^2 takes 20 us; a tile
// kernel (32 x 8 cells staged by tensor copies, flat loops over the staged arrays between block barriers)
// executed 647 thread instructions per cell, 285 of them integer, and took 28.8.
constexpr int kAdjOut = 60;              // output columns of a strip

struct alignas(16) AdjSmem {
    float raw[kAhead][8][64];            // rows in flight: h, z, n, qx, qy of row j; lambda_h, lambda_qx, lambda_qy of row j - 1
    double gn[kAhead][64];               // dL/dn of row j - 2
};

// Two columns of a row.
using Pair = unsigned long long;

__device__ __forceinline__ Pair pair_load(const float *p) { return *reinterpret_cast<const Pair *>(p); }
__device__ __forceinline__ void pair_store(float *p, Pair v) { *reinterpret_cast<Pair *>(p) = v; }
__device__ __forceinline__ float pair_get(Pair v, int k) { return k ? f2unpack(v).y : f2unpack(v).x; }
__device__ __forceinline__ void pair_set(Pair &v, int k, float x)
{
    const float2 p = f2unpack(v);
    v = f2pack(k ? p.x : x, k ? x : p.y);
}
// The lane to the left's second column, the lane to the right's first; the pair one column to the left or right.
__device__ __forceinline__ float pair_from_left(Pair v) { return __shfl_up_sync(0xffffffffu, f2unpack(v).y, 1); }
__device__ __forceinline__ float pair_from_right(Pair v) { return __shfl_down_sync(0xffffffffu, f2unpack(v).x, 1); }
__device__ __forceinline__ Pair pair_right(Pair v) { return f2pack(f2unpack(v).y, pair_from_right(v)); }

// 8 bytes global -> shared, asynchronously (in the thread's current group); in == false: zeros.
__device__ __forceinline__ void copy8(float *dst, const float *src, bool in)
{
    asm volatile("cp.async.ca.shared.global [%0], [%1], 8, %2;" ::"r"((unsigned)__cvta_generic_to_shared(dst)), "l"(src),
                 "r"(in ? 8 : 0)
                 : "memory");
}

// The derivatives of a row's faces.
struct FaceRow {
    Pair q, L, R, n;                     // with respect to the old discharge, the depths of the two cells, n of either
};

__device__ __forceinline__ unsigned long long f2sel(bool x, bool y, unsigned long long a, unsigned long long b)
{
    const float2 u = f2unpack(a), v = f2unpack(b);
    return f2pack(x ? u.x : v.x, y ? u.y : v.y);
}

__device__ __forceinline__ unsigned long long f2rcp(unsigned long long a)
{
    const float2 v = f2unpack(a);
    return f2pack(rcp_fast(v.x), rcp_fast(v.y));
}

// Eq. 3 for two faces (the operations of face_fast_sel, in its order), with what its derivatives
// need.  A dry face is evaluated at depth 1 with a zero reciprocal of its denominator, which makes
// its value and its derivatives zero.
struct Faces2 {
    unsigned long long hs, slope, q, nsum, cr, cq, m, inv, F;   // depth, eta_R - eta_L, old q, n_L + n_R, c r7, c |q| r7,
                                                                // -a1 hs, 1 / den, the new value
};

__device__ __forceinline__ Faces2 faces2_value(unsigned long long hf, unsigned long long slope, unsigned long long q,
                                               unsigned long long nsum, const FastConst &k)
{
    Faces2 f;
    const float2 h0 = f2unpack(hf);
    const bool w0 = h0.x > k.h_dry, w1 = h0.y > k.h_dry;
    const float2 h = make_float2(w0 ? h0.x : 1.0f, w1 ? h0.y : 1.0f);
    f.hs = f2pack(h.x, h.y);
    f.slope = slope;
    f.q = q;
    f.nsum = nsum;
    const float2 l = f2unpack(f2mul(f2pack(lg2_fast(h.x), lg2_fast(h.y)), f2dup(-7.0f / 3.0f)));
    const unsigned long long r7 = f2pack(ex2_fast(l.x), ex2_fast(l.y));
    const unsigned long long c = face_c(nsum, k), cq = face_cq(c, q);
    f.m = f2mul(f2dup(-k.a1), f.hs);
    const float2 rd = f2unpack(f2rcp(f2fma(cq, r7, f2dup(1.0f))));
    f.inv = f2pack(w0 ? rd.x : 0.0f, w1 ? rd.y : 0.0f);
    f.F = f2mul(f2fma(f.m, slope, q), f.inv);
    f.cr = f2mul(c, r7);
    f.cq = f2mul(cq, r7);
    return f;
}

// face_lin's formulas.
__device__ __forceinline__ void faces2_lin(const Faces2 &f, const FastConst &k, unsigned long long &dq, unsigned long long &dL,
                                           unsigned long long &dR, unsigned long long &dn)
{
    // dF/dq = (1 - F c r7 sign(q)) / den, sign(0) = 0
    const float2 qv = f2unpack(f.q), t = f2unpack(f2mul(f.F, f.cr));
    const float t0 = qv.x != 0.0f ? __uint_as_float(__float_as_uint(t.x) ^ (__float_as_uint(qv.x) & 0x80000000u)) : 0.0f;
    const float t1 = qv.y != 0.0f ? __uint_as_float(__float_as_uint(t.y) ^ (__float_as_uint(qv.y) & 0x80000000u)) : 0.0f;
    dq = f2mul(f2sub(f2dup(1.0f), f2pack(t0, t1)), f.inv);
    // dF/dhf, and the explicit dependence on the water levels; max sends hf's part to L on ties
    const unsigned long long Ff = f2mul(f.F, f.cq);
    const unsigned long long dh = f2mul(f2fma(f2mul(Ff, f2dup(7.0f / 3.0f)), f2rcp(f.hs), f2mul(f2dup(-k.a1), f.slope)), f.inv);
    const unsigned long long ex = f2mul(f.m, f.inv);              // minus a1 hf / den
    const float2 sv = f2unpack(f.slope);
    const bool l0 = sv.x <= 0.0f, l1 = sv.y <= 0.0f;
    dL = f2sub(f2sel(l0, l1, dh, 0ull), ex);
    dR = f2add(f2sel(l0, l1, 0ull, dh), ex);
    dn = f2mul(f2mul(Ff, f.inv), f2mul(f2dup(-2.0f), f2rcp(f.nsum)));
}

// a / b: by the reciprocal and its remainder (exact), which leaves less than 2^-21 of a unit in the last place beside the
// rounding, where nothing under- or overflows on the way, else by the division.  An edge strip's chain pays for these two
// at every tick: a sweep of 64 steps of 1024^2 took 2.52 ms so, 2.53 with two divisions, 2.49 with approximate ones.
__device__ __forceinline__ float quotient(float a, float b)
{
    const float y = rcp_fast(b), q = __fmul_rn(a, y);
    const float r = __fmaf_rn(__fmaf_rn(-q, b, a), y, q);
    return fminf(b, fabsf(a)) > 0x1p-60f && fmaxf(b, fabsf(a)) < 0x1p60f ? r : __fdiv_rn(a, b);
}

// A border face of Eq. 5 as a face between the cell (depth h, n) and an outer cell that does not
// exist: its value, and its derivatives with respect to the depth and n of the cell.
__device__ __forceinline__ float border_lin(int type, float inward, float h, float sqrtS, float n, const Geom &G, float inflow,
                                            float &dh, float &dn)
{
    dh = dn = 0.0f;
    if (type == kBcWall) return 0.0f;
    if (type == kBcInflow) return inward * inflow;
    const float q = outflow_fast(h, sqrtS, n, G.dx_f, G.h_dry_f, G.bc_form);
    if (q > 0.0f) {
        dh = quotient(-inward * (G.bc_form == 0 ? 5.0f / 3.0f : 2.0f / 3.0f) * q, h);
        dn = quotient(inward * q, n);
    }
    return -inward * q;
}

__device__ __forceinline__ void adj_rows_item(const AdjArgs<float> &A, const int strip, const int y0, const int y1, AdjSmem &sm)
{
    constexpr int kOut = kAdjOut;
    const StepArgs<float> &a = A.fwd;
    const Geom &G = a.geo;
    const int lane = threadIdx.x;
    const int nx = G.nx, ny = G.ny;
    const size_t P = (size_t)G.pitch;
    const Fwd<float> FW(G, a.ctrl->dt);
    const FastConst Kc = FW.K;
    const int x0 = strip * kOut - 2;
    const int c0 = x0 + 2 * lane;
    const int own_lo = strip * kOut, own_hi = min(own_lo + kOut, nx);
    const bool west = x0 < 0, east = x0 + 63 >= nx;
    const bool in = c0 >= 0 && c0 < (int)P;
    const int jb = max(y0 - 2, 0);
    const int jhi = min(y1 + 1, ny - 1);               // last row of the state
    const int jlast = y1 + 1;                          // last tick: row y1 - 1 is completed
    const int steady_lo = jb > 0 ? jb : 2, steady_hi = nx >= 2 ? jhi : -1;
    const bool full = c0 >= own_lo && c0 + 1 < own_hi;
    const bool part = !full && c0 >= own_lo && (c0 < own_hi || (c0 == nx && own_hi == nx));
    // the border face at x = 0 or x = nx in this lane's columns (with nx < 2 a lane can hold both, and every
    // tick takes the general form); its type, inflow slot and sqrt(S) are read a tick ahead
    const bool lane_w = west && c0 == 0, lane_e = east && nx - c0 >= 0 && nx - c0 < 2;
    const int side = lane_e ? 1 : 0, kb = lane_e ? nx - c0 : lane_w ? 0 : -1;
    int nb_t = kBcWall, nb_s = 0, pb_t = kBcWall, pb_s = 0;
    float nb_q = 0.0f;
    auto border_fetch = [&](int r) {
        if (kb >= 0 && r <= jhi) {
            nb_t = a.bc.type[(side ? ny : 0) + r];
            nb_s = a.bc.slot[(side ? ny : 0) + r];
            nb_q = a.bc.sqrtS_f[(side ? ny : 0) + r];
        }
    };
    border_fetch(jb);
    const size_t lane_off = in ? (size_t)c0 : 0;

    auto issue = [&](int j) {
        float *d = &sm.raw[j & (kAhead - 1)][0][2 * lane];
        if (j <= jhi) {
            const size_t o = (size_t)j * P + lane_off;
            copy8(d, a.h + o, in);
            copy8(d + 64, a.z + o, in);
            copy8(d + 128, a.n + o, in);
            copy8(d + 192, a.qx + o, in);
            copy8(d + 256, a.qy + o, in);
        }
        if (j >= 1 && j <= jlast) {                    // face row ny has lambda_qy only
            const size_t o = (size_t)(j - 1) * P + lane_off;
            if (j - 1 < ny) {
                copy8(d + 320, A.lh + o, in);
                copy8(d + 384, A.lqx + o, in);
            }
            copy8(d + 448, A.lqy + o, in);
        }
        if (j - 2 >= y0 && j - 2 < y1) {
            const double *g = A.gn + (size_t)(j - 2) * P + lane_off;
            copy16(reinterpret_cast<float *>(&sm.gn[j & (kAhead - 1)][2 * lane]), reinterpret_cast<const float *>(g), in);
        }
        copy_commit();
    };
    for (int j = jb; j < jb + kAhead; j++) issue(j);

    // The gauges, from a list in the order of rows, columns and indexes: each lane holds one of a window of 32, with its seed;
    // `pending` are those in the staged cells yet to come, grow the row of the first.  (Crowded items that scanned all gauges at
    // every row took 5.0 ms a step of 1024^2 with 4096 gauges in a 64 x 64 patch, the tile kernel before them 0.76; so 0.092,
    // and 0.019 with one gauge as before.)
    int wx = 0, wrow = 0, wcol = 0, grow = 0x7fffffff;
    float wseed = 0.0f;
    unsigned pending = 0;
    auto window = [&](int x, int row) {                // from x on, or from the first one at (row, x0) or after it
#pragma unroll 1
        for (;;) {
            wx = x;
            const int4 g = x + lane < A.n_gauges ? __ldg(A.gauge_list + x + lane) : make_int4(0x7fffffff, 0, 0, 0);
            const bool mine = g.x >= row && g.x <= jhi && g.y >= x0 && g.y < x0 + 64;
            wrow = g.x;
            wcol = g.y - x0;
            pending = __ballot_sync(0xffffffffu, mine);
            if (pending) {
                wseed = mine ? (float)A.seed[g.z] : 0.0f;
                grow = __shfl_sync(0xffffffffu, wrow, __ffs(pending) - 1);
                return;
            }
            grow = 0x7fffffff;
            const int last = __shfl_sync(0xffffffffu, wrow, 31);
            if (last > jhi) return;
            x = gauge_seek(A.gauge_list, A.n_gauges, x + 32, max(row, last), x0);
        }
    };
    window(A.n_gauges > 32 ? gauge_seek(A.gauge_list, A.n_gauges, 0, jb, x0) : 0, jb);

    Pair hp = 0, zp = 0, np_ = 0;                // row j - 1: depth, bed, n
    Pair xp = 0, yp = 0;                           // its new faces
    FaceRow dx{}, dy{};                                // and their derivatives
    Pair lu2 = 0, acc2 = 0, gx2 = 0, gy2 = 0;  // row j - 2: lu, and its sums so far

    auto tick = [&](auto steady_t, auto edge_t, const int j) {
        constexpr bool kSteady = decltype(steady_t)::value, kEdge = decltype(edge_t)::value;
        const bool row = kSteady || j < ny, rowp = kSteady || (j >= 1 && j <= ny);   // rows j and j - 1 are cells
        copy_wait<kAhead - 1>();
        const float *d = &sm.raw[j & (kAhead - 1)][0][2 * lane];
        const Pair lq = pair_load(d + 384), lqy = pair_load(d + 448);
        Pair lu = pair_load(d + 320);
        double2 gn = *reinterpret_cast<const double2 *>(&sm.gn[j & (kAhead - 1)][2 * lane]);
        Pair ch = 0, cz = 0, cn = 0, cx = 0, cy = 0;
        if (row) {
            ch = pair_load(d);
            cz = pair_load(d + 64);
            cn = pair_load(d + 128);
            cx = pair_load(d + 192);
            cy = pair_load(d + 256);
        }
        issue(j + kAhead);
        // ---- A. the new south faces of row j (their derivatives, and the west faces, after C has used
        // those of row j - 1: they take the same registers)
        const Pair e = f2add(ch, cz);
        const bool inner = kSteady || (j > 0 && j < ny);
        Pair qy = 0, bR = 0, bL = 0, bn = 0;
        Faces2 ya;
        if (inner) {
            const Pair ep = f2add(hp, zp);
            ya = faces2_value(f2sub(f2max(ep, e), f2max(zp, cz)), f2sub(e, ep), cy, f2add(np_, cn), Kc);
            qy = ya.F;
        } else if (j == 0 || j == ny) {
            const int off = j == 0 ? 2 * ny : 2 * ny + nx;
            const Pair hb = j == 0 ? ch : hp, nb = j == 0 ? cn : np_;
#pragma unroll 1
            for (int k = 0; k < 2; k++) {
                const int c = c0 + k;
                if (c < 0 || c >= nx) continue;
                const int t = a.bc.type[off + c];
                float dh, dn;
                const float v = border_lin(t, j == 0 ? 1.0f : -1.0f, pair_get(hb, k), a.bc.sqrtS_f[off + c], pair_get(nb, k), G,
                                           t == kBcInflow ? a.inflow_q[(size_t)a.s * a.n_slots + a.bc.slot[off + c]] : 0.0f,
                                           dh, dn);
                pair_set(qy, k, v);
                if (j == 0) pair_set(bR, k, dh);
                else pair_set(bL, k, dh);
                pair_set(bn, k, dn);
            }
        }
        // ---- B. the adjoint of row j - 1's unclipped depth
        if (rowp) {
            const float2 x01 = f2unpack(xp);
            const float xe = pair_from_right(xp);
            const Pair dv = f2add(f2pack(__fsub_rn(x01.x, x01.y), __fsub_rn(x01.y, xe)), f2sub(yp, qy));
            const float2 u0 = f2unpack(f2fma(f2dup(Kc.dtdx), dv, hp));
            const float u[2] = {u0.x, u0.y};
            float v[2] = {f2unpack(lu).x, f2unpack(lu).y};
            if (grow == j - 1) {                       // the row's seeds, in the list's order (repeated gauges add up in theirs)
#pragma unroll 1
                for (;;) {
                    unsigned now = pending & __ballot_sync(0xffffffffu, wrow == j - 1);
                    pending &= ~now;
#pragma unroll 1
                    for (; now; now &= now - 1) {
                        const int q = __ffs(now) - 1, gc = __shfl_sync(0xffffffffu, wcol, q) - 2 * lane;
                        const float sd = __shfl_sync(0xffffffffu, wseed, q);
#pragma unroll
                        for (int k = 0; k < 2; k++)
                            if (gc == k) v[k] = v[k] + sd;
                    }
                    if (pending) {
                        grow = __shfl_sync(0xffffffffu, wrow, __ffs(pending) - 1);
                        break;
                    }
                    window(wx + 32, j - 1);
                    if (grow != j - 1) break;
                }
            }
#pragma unroll
            for (int k = 0; k < 2; k++) {
                if (u[k] < 0.0f) v[k] = 0.0f;
                if (kEdge && (c0 + k < 0 || c0 + k >= nx)) v[k] = 0.0f;
            }
            lu = f2pack(v[0], v[1]);
        } else {
            lu = 0;
        }
        // ---- C. the x-faces of row j - 1 and the y-faces below it
        const float lul = pair_from_left(lu);
        const float2 a0 = f2unpack(lu);
        const Pair mux = f2fma(f2dup(Kc.dtdx), f2pack(__fsub_rn(a0.x, lul), __fsub_rn(a0.y, a0.x)), lq);
        const Pair muy = f2fma(f2dup(Kc.dtdx), f2sub(lu, lu2), lqy);
        const Pair xL = f2mul(mux, dx.L), xR = f2mul(mux, dx.R), xn = f2mul(mux, dx.n), xq = f2mul(mux, dx.q);
        const Pair yL = f2mul(muy, dy.L), yR = f2mul(muy, dy.R), yn = f2mul(muy, dy.n), yq = f2mul(muy, dy.q);
        const Pair out2 = f2add(acc2, yL), gs2 = f2add(gx2, f2add(gy2, yn));   // row j - 2's sums, complete
        const Pair lu_below = lu2;
        // ---- the rows move on
        acc2 = f2add(f2add(f2add(lu, xR), pair_right(xL)), yR);
        gx2 = f2add(xn, pair_right(xn));
        gy2 = yn;
        lu2 = lu;
        yp = qy;
        const int qb_t = pb_t, qb_s = pb_s;

        if (inner) faces2_lin(ya, Kc, dy.q, dy.L, dy.R, dy.n);
        else dy = FaceRow{0, bL, bR, bn};
        if (row) {
            const float el = pair_from_left(e), zl = pair_from_left(cz), nl = pair_from_left(cn);
            const float2 e0 = f2unpack(e), z0 = f2unpack(cz), n0 = f2unpack(cn);
            const Faces2 xa = faces2_value(f2sub(f2max(f2pack(el, e0.x), e), f2max(f2pack(zl, z0.x), cz)),
                                           f2pack(__fsub_rn(e0.x, el), __fsub_rn(e0.y, e0.x)), cx,
                                           f2pack(__fadd_rn(nl, n0.x), __fadd_rn(n0.x, n0.y)), Kc);
            xp = xa.F;
            faces2_lin(xa, Kc, dx.q, dx.L, dx.R, dx.n);
            if (kEdge && (west || east)) {
                const float hl = pair_from_left(ch);
                // the border face of side sd in this lane's column kf
                auto border = [&](int sd, int t, int slot, float sqrtS) {
                    const int kf = sd ? nx - c0 : 0;
                    const float h = sd && kf == 0 ? hl : f2unpack(ch).x;   // (kf = 1: the cell is the first column)
                    const float n = sd && kf == 0 ? nl : n0.x;
                    float dh, dn;
                    const float v = border_lin(t, sd ? -1.0f : 1.0f, h, sqrtS, n, G,
                                               t == kBcInflow ? a.inflow_q[(size_t)a.s * a.n_slots + slot] : 0.0f, dh, dn);
                    pair_set(xp, kf, v);
                    pair_set(dx.q, kf, 0.0f);
                    pair_set(dx.L, kf, sd ? dh : 0.0f);
                    pair_set(dx.R, kf, sd ? 0.0f : dh);
                    pair_set(dx.n, kf, dn);
                };
                if (kb >= 0) border(side, nb_t, nb_s, nb_q);
                if (!kSteady && lane_w && lane_e) border(0, a.bc.type[j], a.bc.slot[j], a.bc.sqrtS_f[j]);
                pb_t = nb_t;
                pb_s = nb_s;
                border_fetch(j + 1);
            }
        } else {
            xp = 0;
            dx = FaceRow{};
            pb_t = kBcWall;
        }
        hp = ch;
        zp = cz;
        np_ = cn;
        // ---- D. row j - 2 is complete
        if (j - 2 >= y0 && j - 2 < y1) {
            const float2 gs = f2unpack(gs2);
            const size_t o = (size_t)(j - 2) * P + lane_off;
            gn.x += (double)gs.x;
            gn.y += (double)gs.y;
            if (kEdge ? full : lane >= 1 && lane <= kOut / 2) {
                pair_store(A.lh_out + o, out2);
                *reinterpret_cast<double2 *>(A.gn + o) = gn;
            } else if (kEdge && part && c0 < own_hi) {
                A.lh_out[o] = f2unpack(out2).x;
                A.gn[o] = gn.x;
            }
        }
        // the adjoint of the old faces of row j - 1 (and of the grid's north faces, face row ny)
        const int r = j - 1;
        if (r >= y0 && (r < y1 || (r == ny && y1 == ny))) {
            const size_t o = (size_t)r * P + lane_off;
            const bool cells = r < ny;
            if (kEdge ? full : lane >= 1 && lane <= kOut / 2) {
                if (cells) pair_store(A.lqx_out + o, xq);
                pair_store(A.lqy_out + o, yq);
            } else if (kEdge && part) {
#pragma unroll
                for (int k = 0; k < 2; k++) {
                    const int c = c0 + k;
                    if (cells && (c < own_hi || c == nx)) A.lqx_out[o + k] = pair_get(xq, k);
                    if (c < own_hi) A.lqy_out[o + k] = pair_get(yq, k);
                }
            }
            // inflow faces: lu of the cell and lambda_q of the face, for pass 3
            if (A.in_log) {
                if (kEdge && cells && (west || east)) {
                    const int kf = side ? nx - c0 : 0;
                    if (kb >= 0 && qb_t == kBcInflow && (side ? own_hi == nx : own_lo == 0))
                        A.in_log[qb_s] = make_float2(side ? (kf == 0 ? lul : a0.x) : a0.x, pair_get(lq, kf));
                    if (!kSteady && lane_w && lane_e && a.bc.type[r] == kBcInflow)     // nx = 1: the west face too
                        A.in_log[a.bc.slot[r]] = make_float2(a0.x, pair_get(lq, 0));
                }
                if (!kSteady && (r == 0 || r == ny)) {
                    const int off = r == 0 ? 2 * ny : 2 * ny + nx;
                    const Pair lb = r == 0 ? lu : lu_below;
#pragma unroll
                    for (int k = 0; k < 2; k++) {
                        const int c = c0 + k;
                        if (c >= own_lo && c < own_hi && a.bc.type[off + c] == kBcInflow)
                            A.in_log[a.bc.slot[off + c]] = make_float2(pair_get(lb, k), pair_get(lqy, k));
                    }
                }
            }
        }
    };

    int j = jb;
    if (jb > 0) {                                      // row y0 - 2 is only the row below
        copy_wait<kAhead - 1>();
        const float *d = &sm.raw[jb & (kAhead - 1)][0][2 * lane];
        hp = pair_load(d);
        zp = pair_load(d + 64);
        np_ = pair_load(d + 128);
        border_fetch(jb + 1);
        issue(jb + kAhead);
        j++;
    }
    while (j <= jlast) {
        if (j >= steady_lo && j <= steady_hi) {
            if (west || east) {
#pragma unroll 1
                for (; j <= steady_hi; j++) tick(std::true_type{}, std::true_type{}, j);
            } else {
#pragma unroll 1
                for (; j <= steady_hi; j++) tick(std::true_type{}, std::false_type{}, j);
            }
        } else {
            const int e = j < steady_lo ? min(jlast, steady_lo - 1) : jlast;
#pragma unroll 1
            for (; j <= e; j++) tick(std::false_type{}, std::true_type{}, j);
        }
    }
    copy_wait<0>();
}

__global__ void __launch_bounds__(32, 12) adj_rows_kernel(const __grid_constant__ AdjArgs<float> A, const int rows, const int rows_edge)
{
    __shared__ AdjSmem sm;
    pdl_wait();
    pdl_launch();
    constexpr int kOut = kAdjOut;
    const int n_strips = (A.fwd.geo.nx + kOut - 1) / kOut, n_edge = min(n_strips, 2);
    const int edge_items = n_edge * ((A.fwd.geo.ny + rows_edge - 1) / rows_edge), item = blockIdx.x;
    int strip, y0, r;
    if (item < edge_items) {
        strip = item % n_edge ? n_strips - 1 : 0;
        r = rows_edge;
        y0 = (item / n_edge) * r;
    } else {
        strip = 1 + (item - edge_items) % (n_strips - n_edge);
        r = rows;
        y0 = (item - edge_items) / (n_strips - n_edge) * r;
    }
    adj_rows_item(A, strip, y0, min(y0 + r, A.fwd.geo.ny), sm);
}

// Pass 3 over the logged steps, block (entry, section): the formulas of inflow_adjoint on the logged lu
// and lambda_q, each section cell's term into the entry's row of A.terms.
__global__ void __launch_bounds__(64) adj_inflow_terms_kernel(const AdjInflowArgs A)
{
    __shared__ double red[32];
    const int e = blockIdx.x, tid = threadIdx.x;
    const InflowSec S = A.secs[blockIdx.y];
    const int64_t step = A.first_step - e;           // global step of the entry
    const int64_t ie = step / A.E - A.e0;
    const int s = (int)(step % A.E);
    const double Q = A.inflow_Q[ie * A.nQ + (size_t)s * A.n_sec + blockIdx.y];
    const double W = A.inflow_W[ie * A.nQ + (size_t)s * A.n_sec + blockIdx.y];
    const float *iq = A.inflow_q + ((size_t)ie * A.E + s) * A.n_slots;
    const float2 *log = A.log + (size_t)e * A.n_slots;
    double *terms = A.terms + (size_t)e * A.n_slots;
    const double dx = A.geo.dx, dtdx = A.dt[ie] / A.geo.dx;
    const double pe = A.geo.bc_form == 0 ? 5.0 / 3.0 : 2.0 / 3.0;
    const double inward = (double)inward_sign(S.side);
    auto nu_of = [&](int c) {
        const float2 v = log[S.slot0 + c];
        return inward * ((double)v.y + inward * dtdx * (double)v.x) / dx;
    };
    double D = 0.0, N = 0.0;
    if (Q > 0.0)
        for (int c = tid; c < S.ncell; c += 64) {
            const double hh = W - (double)A.z[A.cells[S.cell0 + c]];
            if (!(hh > 0.0)) continue;
            const double k = pe * ((double)iq[S.slot0 + c] * dx) / hh;
            D += k;
            N += nu_of(c) * k;
        }
    D = block_reduce<false>(D, red);
    __syncthreads();
    if (tid == 0) red[31] = D;
    __syncthreads();
    D = red[31];
    __syncthreads();
    N = block_reduce<false>(N, red);
    __syncthreads();
    if (tid == 0) red[30] = N;
    __syncthreads();
    N = red[30];
    for (int c = tid; c < S.ncell; c += 64) {
        const int64_t idx = A.cells[S.cell0 + c];
        const double hh = W - (double)A.z[idx];
        double t = 0.0;
        if (Q > 0.0 && D > 0.0 && hh > 0.0) t = ((double)iq[S.slot0 + c] * dx / (double)A.n[idx]) * (N / D - nu_of(c));
        terms[S.slot0 + c] = t;
    }
}

// Each section cell's terms, in the order of the sweep.
__global__ void adj_inflow_sum_kernel(const AdjInflowArgs A)
{
    const int c = blockIdx.x * blockDim.x + threadIdx.x;
    if (c >= A.n_slots) return;
    double g = A.gn_in[c];
    for (int e = 0; e < A.n_entries; e++) g += A.terms[(size_t)e * A.n_slots + c];
    A.gn_in[c] = g;
}

// ---------------------------------------------------------------- the scheme options
// With the theta weighting or the vector norm a face's new value also depends
// on its two neighbours along the axis and on the four faces of the other axis
// around it, so their adjoints receive contributions too.  The reverse step
// then runs in three passes over global memory (each face's derivatives once):
//  R1 per cell: the new faces (the forward kernels' own arithmetic, so the clip
//     and wet/dry decisions are the forward's), the clip mask, and the adjoint
//     of the unclipped depth (gauge seeds added by a one-thread pass after it);
//  R2 per face: mu and the face's derivatives, stored as its contributions to
//     the two cells (depth, Manning n), to its own old discharge, to its axis
//     neighbours (theta) and to the orthogonal faces (vector norm);
//  R3 per cell: the gathers, for the cell and for the faces it owns (its west
//     and south faces; the last column and row also the east and north ones).
// Scratch planes (pitch x (ny + 1) each): 0..4 x-faces (to L, to R, dL/dn,
// to the axis neighbours, to the orthogonal faces), 5..9 the same for y-faces,
// 10 the clip mask.
template <typename T> struct OptFace;

template <> struct OptFace<float> {
    FastConst K;
    __device__ OptFace(const Geom &G, double dt_)
    {
        const float dt = (float)dt_, dx = (float)G.dx;
        K.gdt = (float)G.g * dt;
        K.a1 = K.gdt / dx;
        K.gdt4 = 0.25f * K.gdt;
        K.h_dry = (float)G.h_dry;
        K.dtdx = dt / dx;
        K.theta = (float)G.theta;
        K.w = (float)(0.5 * (1.0 - G.theta));
    }
    __device__ float qn(float q, float qp, float qx, bool th) const { return th ? theta_q(q, qp, qx, K) : q; }
    __device__ float qm(float q, float a, float b, float c, float d, bool vec) const
    {
        return vec ? q_norm(q, a, b, c, d) : fabsf(q);
    }
    __device__ float qo(float a, float b, float c, float d) const
    {
        return __fmul_rn(0.25f, __fadd_rn(__fadd_rn(a, b), __fadd_rn(c, d)));
    }
    __device__ float face(float qmag, float qnum, float hL, float zL, float nL, float hR, float zR, float nR) const
    {
        return face_fast_gen(qmag, qnum, hL + zL, hR + zR, fmaxf(zL, zR), nL + nR, K);
    }
};

template <> struct OptFace<double> {
    double g, dt, hd, th, w;
    Divisor<double> over_dx;
    __device__ OptFace(const Geom &G, double dt_)
        : g(G.g), dt(dt_), hd(G.h_dry), th(G.theta), w(0.5 * (1.0 - G.theta)), over_dx(G.dx) {}
    __device__ double qn(double q, double qp, double qx, bool t) const { return theta_q_ieee<double>(q, qp, qx, th, w, t); }
    __device__ double qm(double q, double a, double b, double c, double d, bool vec) const
    {
        return q_norm_ieee<double>(q, a, b, c, d, vec);
    }
    __device__ double qo(double a, double b, double c, double d) const
    {
        using O = R<double>;
        return O::mul(0.25, O::add(O::add(a, b), O::add(c, d)));
    }
    __device__ double face(double qmag, double qnum, double hL, double zL, double nL, double hR, double zR,
                           double nR) const
    {
        return face_update_ieee<double>(qnum, qmag, hL, zL, nL, hR, zR, nR, g, dt, over_dx, hd);
    }
};

// Inputs of an interior face: its old q, the numerator discharge, the friction
// magnitude and the mean orthogonal discharge, with the forward step's neighbours.
template <typename T>
struct OptIn {
    T q, qn, qm, qo;
};

template <typename T>
__device__ __forceinline__ OptIn<T> opt_x_in(const StepArgs<T> &a, const OptFace<T> &O, int j, int fi, bool th,
                                             bool vec)
{
    const size_t P = (size_t)a.geo.pitch, r = (size_t)j * P;
    OptIn<T> v;
    v.q = a.qx[r + fi];
    v.qn = O.qn(v.q, a.qx[r + fi - 1], a.qx[r + fi + 1], th);
    const T qa = a.qy[r + fi - 1], qb = a.qy[r + fi], qc = a.qy[r + P + fi - 1], qd = a.qy[r + P + fi];
    v.qm = O.qm(v.q, qa, qb, qc, qd, vec);
    v.qo = vec ? O.qo(qa, qb, qc, qd) : T(0);
    return v;
}

template <typename T>
__device__ __forceinline__ OptIn<T> opt_y_in(const StepArgs<T> &a, const OptFace<T> &O, int fj, int i, bool th,
                                             bool vec)
{
    const size_t P = (size_t)a.geo.pitch, r = (size_t)fj * P;
    OptIn<T> v;
    v.q = a.qy[r + i];
    v.qn = O.qn(v.q, a.qy[r - P + i], a.qy[r + P + i], th);
    const T qa = a.qx[r - P + i], qb = a.qx[r - P + i + 1], qc = a.qx[r + i], qd = a.qx[r + i + 1];
    v.qm = O.qm(v.q, qa, qb, qc, qd, vec);
    v.qo = vec ? O.qo(qa, qb, qc, qd) : T(0);
    return v;
}

// New value of x-face (j, fi), fi in [0, nx], and of y-face (fj, i), fj in [0, ny].
template <typename T>
__device__ __forceinline__ T opt_new_x(const StepArgs<T> &a, const Fwd<T> &F, const OptFace<T> &O, int j, int fi,
                                       bool th, bool vec)
{
    const Geom &G = a.geo;
    const size_t r = (size_t)j * G.pitch;
    if (fi == 0) return bface(a, F, 0, j, a.h[r], a.n[r]);
    if (fi == G.nx) return bface(a, F, 1, j, a.h[r + G.nx - 1], a.n[r + G.nx - 1]);
    const OptIn<T> v = opt_x_in(a, O, j, fi, th, vec);
    return O.face(v.qm, v.qn, a.h[r + fi - 1], a.z[r + fi - 1], a.n[r + fi - 1], a.h[r + fi], a.z[r + fi], a.n[r + fi]);
}

template <typename T>
__device__ __forceinline__ T opt_new_y(const StepArgs<T> &a, const Fwd<T> &F, const OptFace<T> &O, int fj, int i,
                                       bool th, bool vec)
{
    const Geom &G = a.geo;
    const size_t P = (size_t)G.pitch, r = (size_t)fj * P;
    if (fj == 0) return bface(a, F, 2, i, a.h[i], a.n[i]);
    if (fj == G.ny) return bface(a, F, 3, i, a.h[r - P + i], a.n[r - P + i]);
    const OptIn<T> v = opt_y_in(a, O, fj, i, th, vec);
    return O.face(v.qm, v.qn, a.h[r - P + i], a.z[r - P + i], a.n[r - P + i], a.h[r + i], a.z[r + i], a.n[r + i]);
}

// Derivatives of one wet face F = (qn - a1 hf (eta_R - eta_L)) / (1 + cc qmag),
// cc = g dt nf^2 hf^(-7/3): own old q, each axis neighbour (theta), each of
// the four orthogonal faces (vector norm), h_L, h_R and n (per cell).
template <typename T> struct OptLin {
    T dq, dnb, dorth, dhL, dhR, dn;
};

template <typename T>
__device__ __forceinline__ OptLin<T> opt_lin(const OptIn<T> &v, T hL, T zL, T nL, T hR, T zR, T nR, T hf, T g, T dt,
                                             T dx, T th, T w, bool vec)
{
    OptLin<T> r;
    const T etaL = hL + zL, etaR = hR + zR;
    const T nf = T(0.5) * (nL + nR);
    const T gdt = g * dt, a1 = gdt / dx;
    const T cc = gdt * nf * nf * Fwd<T>::pow_m73_(hf);
    const T fric = cc * v.qm;
    const T inv_den = Fwd<T>::rcp_(T(1) + fric);
    const T F = (v.qn - a1 * hf * (etaR - etaL)) * inv_den;
    const T dF_dqm = -F * cc * inv_den;
    T dqm_dq, dqm_dqo;
    if (!vec) {
        dqm_dq = v.q > T(0) ? T(1) : (v.q < T(0) ? T(-1) : T(0));
        dqm_dqo = T(0);
    } else if (v.qm > T(0)) {
        const T inv = Fwd<T>::rcp_(v.qm);
        dqm_dq = v.q * inv;
        dqm_dqo = v.qo * inv;
    } else {
        dqm_dq = dqm_dqo = T(0);
    }
    r.dq = th * inv_den + dF_dqm * dqm_dq;
    r.dnb = w * inv_den;
    r.dorth = T(0.25) * dF_dqm * dqm_dqo;
    const T dF_dhf = (-a1 * (etaR - etaL) + F * (T(7) / T(3)) * fric * Fwd<T>::rcp_(hf)) * inv_den;
    const T d_expl = a1 * hf * inv_den;
    const bool left = etaL >= etaR;
    r.dhL = d_expl + (left ? dF_dhf : T(0));
    r.dhR = -d_expl + (left ? T(0) : dF_dhf);
    r.dn = -F * fric * inv_den * Fwd<T>::rcp_(nf);
    return r;
}

template <typename T>
__device__ __forceinline__ T *opt_plane(const AdjArgs<T> &A, int k)
{
    return A.scratch + (size_t)k * A.fwd.geo.pitch * (A.fwd.geo.ny + 1);
}

// R1: clip mask and the adjoint of the unclipped depth of every cell.
template <typename T>
__global__ void __launch_bounds__(256) adj_opt_cells_kernel(const AdjArgs<T> A, const int nbx)
{
    const StepArgs<T> &a = A.fwd;
    const Geom &G = a.geo;
    const int i = (int)(blockIdx.x % (unsigned)nbx) * BX + threadIdx.x;
    const int j = (int)(blockIdx.x / (unsigned)nbx) * 8 + threadIdx.y;
    if (i >= G.nx || j >= G.ny) return;
    const bool th = G.theta != 1.0, vec = G.friction != 0;
    const Fwd<T> F(G, a.ctrl->dt);
    const OptFace<T> O(G, a.ctrl->dt);
    const size_t c = (size_t)j * G.pitch + i;
    const T qW = opt_new_x(a, F, O, j, i, th, vec), qE = opt_new_x(a, F, O, j, i + 1, th, vec);
    const T qS = opt_new_y(a, F, O, j, i, th, vec), qN = opt_new_y(a, F, O, j + 1, i, th, vec);
    const T hu = F.update(a.h[c], qW, qE, qS, qN);
    const bool keep = !(hu < T(0));
    A.lhu[c] = keep ? A.lh[c] : T(0);
    opt_plane(A, 10)[c] = keep ? T(1) : T(0);
}

// Gauge seeds into the unclipped depth's adjoint, in gauge order (repeated gauges add up in order).
template <typename T>
__global__ void adj_opt_seeds_kernel(const AdjArgs<T> A)
{
    if (threadIdx.x != 0 || blockIdx.x != 0) return;
    const Geom &G = A.fwd.geo;
    for (int k = 0; k < A.n_gauges; k++) {
        const int64_t flat = A.gauge_cells[k];
        const size_t c = (size_t)(flat / G.nx) * G.pitch + (size_t)(flat % G.nx);
        if (opt_plane(A, 10)[c] != T(0)) A.lhu[c] = A.lhu[c] + T(A.seed[k]);
    }
}

// R2: every face's contributions (axis 0: x-faces, rows ny, faces nx + 1; axis 1: y-faces).
template <typename T>
__global__ void __launch_bounds__(256) adj_opt_faces_kernel(const AdjArgs<T> A, const int axis, const int nbx)
{
    const StepArgs<T> &a = A.fwd;
    const Geom &G = a.geo;
    const int nx = G.nx, ny = G.ny;
    const int fi = (int)(blockIdx.x % (unsigned)nbx) * BX + threadIdx.x;
    const int fj = (int)(blockIdx.x / (unsigned)nbx) * 8 + threadIdx.y;
    const int ncol = axis == 0 ? nx + 1 : nx, nrow = axis == 0 ? ny : ny + 1;
    if (fi >= ncol || fj >= nrow) return;
    const bool th = G.theta != 1.0, vec = G.friction != 0;
    const Fwd<T> F(G, a.ctrl->dt);
    const OptFace<T> O(G, a.ctrl->dt);
    const T dt = T(a.ctrl->dt), dx = T(G.dx), g = T(G.g), hd = T(G.h_dry), dtdx = dt / dx;
    const T tw = T(G.theta), ww = T(0.5 * (1.0 - G.theta));
    const size_t P = (size_t)G.pitch, f = (size_t)fj * P + fi;
    // the face's two cells (L lower index, R) as flat pitched indices, and whether they exist
    const bool hasL = axis == 0 ? fi > 0 : fj > 0, hasR = axis == 0 ? fi < nx : fj < ny;
    const size_t cL = axis == 0 ? f - 1 : f - P, cR = f;
    const T lL = hasL ? A.lhu[cL] : T(0), lR = hasR ? A.lhu[cR] : T(0);
    const T mu = (axis == 0 ? A.lqx[f] : A.lqy[f]) + dtdx * (lR - lL);
    T cl = T(0), cr = T(0), cn = T(0), lq = T(0), lt = T(0), lo = T(0);
    if (!hasL || !hasR) {                                    // a border face: Eq. 5-6 or a wall
        const int side = axis == 0 ? (hasL ? 1 : 0) : (hasL ? 3 : 2);
        const int k = axis == 0 ? fj : fi;
        const size_t cell = hasL ? cL : cR;
        outflow_adj(a, F, side, k, a.h[cell], a.n[cell], mu, hasL ? cl : cr, cn);
    } else {
        const OptIn<T> v = axis == 0 ? opt_x_in(a, O, fj, fi, th, vec) : opt_y_in(a, O, fj, fi, th, vec);
        const T hL = a.h[cL], zL = a.z[cL], nL = a.n[cL], hR = a.h[cR], zR = a.z[cR], nR = a.n[cR];
        const T hf = F.hf(hL, zL, hR, zR);
        if (hf > hd && mu != T(0)) {
            const OptLin<T> d = opt_lin<T>(v, hL, zL, nL, hR, zR, nR, hf, g, dt, dx, tw, ww, vec);
            cl = mu * d.dhL;
            cr = mu * d.dhR;
            cn = mu * d.dn;
            lq = mu * d.dq;
            lt = th ? mu * d.dnb : T(0);
            lo = vec ? mu * d.dorth : T(0);
        }
    }
    const int b = axis == 0 ? 0 : 5;
    opt_plane(A, b + 0)[f] = cl;
    opt_plane(A, b + 1)[f] = cr;
    opt_plane(A, b + 2)[f] = cn;
    opt_plane(A, b + 3)[f] = lt;
    opt_plane(A, b + 4)[f] = lo;
    (axis == 0 ? A.lqx_out : A.lqy_out)[f] = lq;
}

// R3: per cell, its own adjoint and dL/dn, and the gathers of the faces it owns.
template <typename T>
__global__ void __launch_bounds__(256) adj_opt_gather_kernel(const AdjArgs<T> A, const int nbx)
{
    const Geom &G = A.fwd.geo;
    const int nx = G.nx, ny = G.ny;
    const int i = (int)(blockIdx.x % (unsigned)nbx) * BX + threadIdx.x;
    const int j = (int)(blockIdx.x / (unsigned)nbx) * 8 + threadIdx.y;
    if (i >= nx || j >= ny) return;
    const size_t P = (size_t)G.pitch, c = (size_t)j * P + i;
    const T *XL = opt_plane(A, 0), *XR = opt_plane(A, 1), *XN = opt_plane(A, 2), *XT = opt_plane(A, 3),
            *XO = opt_plane(A, 4);
    const T *YL = opt_plane(A, 5), *YR = opt_plane(A, 6), *YN = opt_plane(A, 7), *YT = opt_plane(A, 8),
            *YO = opt_plane(A, 9);
    A.lh_out[c] = A.lhu[c] + XR[c] + XL[c + 1] + YR[c] + YL[c + P];
    const T gs = (XN[c] + XN[c + 1]) + (YN[c] + YN[c + P]);
    A.gn[c] += (double)gs;
    // x-face (j, fi): theta from x-faces fi - 1 and fi + 1; vector norm from the y-faces
    // (j, fi - 1), (j, fi), (j + 1, fi - 1), (j + 1, fi) that read its old value
    auto gather_x = [&](int fi) {
        const size_t f = (size_t)j * P + fi;
        T s = T(0);
        if (fi > 0) s += XT[f - 1];
        if (fi < nx) s += XT[f + 1];
        if (fi > 0) s += YO[f - 1] + YO[f + P - 1];
        if (fi < nx) s += YO[f] + YO[f + P];
        A.lqx_out[f] += s;
    };
    // y-face (fj, i): theta from y-faces fj - 1 and fj + 1; vector norm from the x-faces
    // (fj - 1, i), (fj - 1, i + 1), (fj, i), (fj, i + 1) that read its old value
    auto gather_y = [&](int fj) {
        const size_t f = (size_t)fj * P + i;
        T s = T(0);
        if (fj > 0) s += YT[f - P];
        if (fj < ny) s += YT[f + P];
        if (fj > 0) s += XO[f - P] + XO[f - P + 1];
        if (fj < ny) s += XO[f] + XO[f + 1];
        A.lqy_out[f] += s;
    };
    gather_x(i);
    if (i == nx - 1) gather_x(nx);
    gather_y(j);
    if (j == ny - 1) gather_y(ny);
}

template <typename T>
__global__ void gn_out_kernel(Geom G, const double *gn, T *dst)
{
    const size_t N = (size_t)G.nx * G.ny;
    for (size_t k = blockIdx.x * (size_t)blockDim.x + threadIdx.x; k < N; k += (size_t)gridDim.x * blockDim.x) {
        const size_t c = (k / G.nx) * G.pitch + k % G.nx;
        dst[c] = T(gn[c]);
    }
}

}  // namespace

template <typename T>
cudaError_t launch_gn_out(const Geom &g, const double *gn, T *dst, cudaStream_t st)
{
    const size_t N = (size_t)g.nx * g.ny;
    const int blocks = (int)std::min<size_t>((N + 255) / 256, 152 * 16);
    gn_out_kernel<T><<<blocks, 256, 0, st>>>(g, gn, dst);
    return cudaGetLastError();
}

template cudaError_t launch_gn_out<float>(const Geom &, const double *, float *, cudaStream_t);

namespace {
// One block, section by section: a corner cell may belong to several, a cell to a section only once.
__global__ void __launch_bounds__(256) gn_inflow_add_kernel(double *gn, const double *gn_in, const InflowSec *secs, const int64_t *cells,
                                                            int n_sec)
{
    for (int k = 0; k < n_sec; k++) {
        const InflowSec S = secs[k];
        for (int c = threadIdx.x; c < S.ncell; c += 256) gn[cells[S.cell0 + c]] += gn_in[S.slot0 + c];
        __syncthreads();
    }
}
}  // namespace

cudaError_t launch_gn_inflow_add(double *gn, const double *gn_in, const InflowSec *secs, const int64_t *sec_cells, int n_sec,
                                 cudaStream_t st)
{
    if (n_sec <= 0) return cudaSuccess;
    gn_inflow_add_kernel<<<1, 256, 0, st>>>(gn, gn_in, secs, sec_cells, n_sec);
    return cudaGetLastError();
}
template cudaError_t launch_gn_out<double>(const Geom &, const double *, double *, cudaStream_t);

template <typename T>
cudaError_t launch_adjoint_step(const AdjArgs<T> &A, cudaStream_t st)
{
    const Geom &G = A.fwd.geo;
    if (G.theta != 1.0 || G.friction != 0) {
        if (!A.scratch) return cudaErrorInvalidValue;
        const dim3 block(BX, 8);
        const int nbx = (G.nx + BX - 1) / BX, nby = (G.ny + 7) / 8;
        adj_opt_cells_kernel<T><<<(unsigned)((int64_t)nbx * nby), block, 0, st>>>(A, nbx);
        if (A.n_gauges > 0) adj_opt_seeds_kernel<T><<<1, 32, 0, st>>>(A);
        const int nbx0 = (G.nx + 1 + BX - 1) / BX;
        adj_opt_faces_kernel<T><<<(unsigned)((int64_t)nbx0 * nby), block, 0, st>>>(A, 0, nbx0);
        const int nby1 = (G.ny + 1 + 7) / 8;
        adj_opt_faces_kernel<T><<<(unsigned)((int64_t)nbx * nby1), block, 0, st>>>(A, 1, nbx);
        adj_opt_gather_kernel<T><<<(unsigned)((int64_t)nbx * nby), block, 0, st>>>(A, nbx);
    } else if constexpr (std::is_same<T, float>::value) {
        int rows = 0, edge = 0;
        // (an item runs three ticks more than it has rows)
        tiled_rows_for((G.nx + kAdjOut - 1) / kAdjOut, G.ny, 3, 12, 900.0, 350.0, 500.0, &rows, &edge);
        const int items = tiled_item_count(G.nx, G.ny, kAdjOut, rows, edge);
        return launch_pdl(adj_rows_kernel, items, 32, st, A, rows, edge);   // pass 3: launch_adjoint_inflow, after the steps
    } else {
        constexpr int BYT = TileRows<T>::v;
        dim3 block(BX, BYT);
        const int nbx = (G.nx + BX - 1) / BX, nby = (G.ny + BYT - 1) / BYT;
        adj_step_kernel<T><<<(unsigned)((int64_t)nbx * nby), block, 0, st>>>(A, nbx);
    }
    if (A.fwd.n_inflow_sec > 0) adj_inflow_kernel<T><<<A.fwd.n_inflow_sec, 256, 0, st>>>(A);
    return cudaGetLastError();
}

cudaError_t launch_adjoint_inflow(const AdjInflowArgs &A, cudaStream_t st)
{
    if (A.n_entries <= 0 || A.n_sec <= 0) return cudaSuccess;
    adj_inflow_terms_kernel<<<dim3(A.n_entries, A.n_sec), 64, 0, st>>>(A);
    adj_inflow_sum_kernel<<<(A.n_slots + 63) / 64, 64, 0, st>>>(A);
    return cudaGetLastError();
}

template cudaError_t launch_adjoint_step<float>(const AdjArgs<float> &, cudaStream_t);
template cudaError_t launch_adjoint_step<double>(const AdjArgs<double> &, cudaStream_t);

}  // namespace flood
