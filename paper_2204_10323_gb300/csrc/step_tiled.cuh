// step_tiled.cuh -- FP32 temporal blocking: one warp advances a strip of columns
// by K <= 4 time steps per launch, with the state of every time level in
// registers.  step_tiled.cu instantiates Eq. 3 as printed and step_tiled_opts.cu
// the scheme options (theta weighting, vector-norm friction).
//
// A work item is a strip of 120 output columns (128 staged, four per lane; the
// halo columns lie in lanes 0 and 31) and a chunk of rows; one 32-thread block
// runs one item, so the hardware's block scheduler hands the items out as warps
// come free.  The warp walks its rows south to north.  At tick j, time level s
// (s = 1 .. K) has row r = j - (s - 1) before it: it computes the new south
// faces of row r, finishes row r - 1 (Eq. 4) and computes the new west faces of
// row r.  Level 1 reads row j of the old state from shared memory, where it
// arrived by asynchronous copies two ticks ahead; level s > 1 takes the row that
// level s - 1 finished in the same tick, in registers; level K stores.  Each
// level keeps one row (old depth, new west and south faces: 12 registers), so no
// level waits for another warp and nothing is handed over through memory.  A
// lane's shared memory holds only its own four columns: no barrier is needed.
// The dependency cone of K steps is K columns wide on each side and K rows at
// each end of a chunk: an item runs 2K ticks more than it has rows.
//
// What bounds it: instruction issue.  At 16384^2 a launch of 4 steps executes
// 1.44 warp instructions per cell-update and moves 8.1 B of DRAM traffic per
// cell-update.  A pipeline of K warps per strip with the rows handed over through
// shared memory and a barrier per tick, two z and n loads and a Manning factor
// per level, executed 3.4.
//
// Per cell and level the arithmetic is the single-step kernels' (the same
// explicitly rounded face function and depth update, two faces per paired
// instruction), so K levels give the same bits as K single steps.  Border faces
// (Eq. 5-6) use that level's inflow row; ledger volumes are booked only by the
// item that owns the cell or border face.
#pragma once

#include <type_traits>

#include "fast_face.cuh"
#include "pdl.cuh"

namespace flood {

// Rows per work item and pipelines for `resident` pipelines that walk the items in turn.
void tiled_split_dynamic(int n_strips, int ny, int resident, int K, int *chunk_rows, int *blocks);

// halo columns per side (at least K: the dependency cone of K steps) and
// output columns of a 128-column strip, per steps per launch K
__host__ __device__ constexpr int halo_cols(int K) { return K <= 4 ? 4 : 8; }
// Right-hand halo: the theta weighting of the strip's last face needs the face
// beyond the staged columns, so with it the cone reaches one column further on
// that side (K + 1 columns after K levels); the left edge loses nothing more.
// Rounded up to a multiple of 4 columns: a strip's first column x0 must stay
// a multiple of 4 (16-byte aligned copies and stores).
__host__ __device__ constexpr int halo_right(int K, int mode)
{
    return (mode & 1) && K + 1 > halo_cols(K) ? (K + 1 + 3) / 4 * 4 : halo_cols(K);
}
__host__ __device__ constexpr int out_cols(int K, int mode = 0) { return 128 - halo_cols(K) - halo_right(K, mode); }
static_assert(out_cols(4, 1) == 116 && out_cols(4, 2) == 120, "strip widths");
static_assert(out_cols(1, 1) % 4 == 0 && out_cols(2, 1) % 4 == 0 && out_cols(3, 1) % 4 == 0 && out_cols(4, 1) % 4 == 0 &&
                  halo_cols(4) % 4 == 0,
              "strip origins must stay multiples of 4 columns");

// Items resident per SM that the launch bounds ask for: 8, 12 or 16 (255, 168 or 128 registers; the
// compiler knows no steps between).  Gcell/s at 12 / 16, Eq. 3 as printed, 16384^2: 577 / 563 (16 spills
// 176 bytes).  At 12 / 8, vector norm, 8192^2: 414 / 393 (12 spilled 200 bytes then, 48 now, and leads); theta,
// 8192^2: 424 / 434 and 1500 x 701: 100 / 111.
__host__ __device__ constexpr int tiled_warps(int mode) { return (mode & 1) ? 8 : 12; }

// Items of a grid for `rows` and `rows_edge` rows per item, the edge strips' first (they take
// the longest, and the tail of a launch is the shorter for it).
__host__ __device__ inline int tiled_item_count(int nx, int ny, int out, int rows, int rows_edge)
{
    const int n_strips = (nx + out - 1) / out, n_edge = n_strips < 2 ? n_strips : 2;
    return n_edge * ((ny + rows_edge - 1) / rows_edge) + (n_strips - n_edge) * ((ny + rows - 1) / rows);
}

namespace {

// Four columns of one row as two packed pairs, in the order of a 16-byte load.
struct Row4 {
    unsigned long long a, b;
};

__device__ __forceinline__ Row4 row_load(const float *p)
{
    const ulonglong2 v = *reinterpret_cast<const ulonglong2 *>(p);
    return Row4{v.x, v.y};
}

__device__ __forceinline__ void row_store(float *p, const Row4 &v)
{
    *reinterpret_cast<ulonglong2 *>(p) = make_ulonglong2(v.a, v.b);
}

__device__ __forceinline__ float row_get(const Row4 &v, int k)
{
    const float2 p = f2unpack(k < 2 ? v.a : v.b);
    return (k & 1) ? p.y : p.x;
}

__device__ __forceinline__ Row4 row_pack(float x, float y, float z, float w) { return Row4{f2pack(x, y), f2pack(z, w)}; }

// The row one column to the left (`left`: the column before the first) or to the right.
__device__ __forceinline__ Row4 row_left(const Row4 &v, float left)
{
    const float2 a = f2unpack(v.a), b = f2unpack(v.b);
    return row_pack(left, a.x, a.y, b.x);
}

__device__ __forceinline__ Row4 row_right(const Row4 &v, float right)
{
    const float2 a = f2unpack(v.a), b = f2unpack(v.b);
    return row_pack(a.y, b.x, b.y, right);
}

// The lane to the left's last column, the lane to the right's first.
__device__ __forceinline__ float from_left(const Row4 &v) { return __shfl_up_sync(0xffffffffu, f2unpack(v.b).y, 1); }
__device__ __forceinline__ float from_right(const Row4 &v) { return __shfl_down_sync(0xffffffffu, f2unpack(v.a).x, 1); }

// max that keeps a NaN
__device__ __forceinline__ float max_nan(float a, float b)
{
    float r;
    asm("max.NaN.f32 %0, %1, %2;" : "=f"(r) : "f"(a), "f"(b));
    return r;
}

__device__ __forceinline__ unsigned long long f2dup(float v) { return f2pack(v, v); }

__device__ __forceinline__ unsigned long long f2max(unsigned long long a, unsigned long long b)
{
    const float2 x = f2unpack(a), y = f2unpack(b);
    return f2pack(fmaxf(x.x, y.x), fmaxf(x.y, y.y));
}

// c = (g dt / 4)(n_L + n_R)^2 of two faces from the sums of their cells' Manning n
__device__ __forceinline__ unsigned long long face_c(unsigned long long nsum, const FastConst &k)
{
    return f2mul(f2dup(k.gdt4), f2mul(nsum, nsum));
}

// c |q| of two faces
__device__ __forceinline__ unsigned long long face_cq(unsigned long long c, unsigned long long q)
{
    const float2 cv = f2unpack(c), qv = f2unpack(q);
    return f2pack(__fmul_rn(cv.x, fabsf(qv.x)), __fmul_rn(cv.y, fabsf(qv.y)));
}

// Eq. 3 for two faces given the flow depth, eta_R - eta_L, the numerator discharge and
// cq = c |q|: the operations of face_fast_sel_gen, in its order.
__device__ __forceinline__ unsigned long long faces2(unsigned long long hf, unsigned long long slope,
                                                     unsigned long long qn, unsigned long long cq, const FastConst &k)
{
    const float2 h = f2unpack(hf);
    const float2 l = f2unpack(f2mul(f2pack(lg2_fast(h.x), lg2_fast(h.y)), f2dup(-7.0f / 3.0f)));
    const unsigned long long r7 = f2pack(ex2_fast(l.x), ex2_fast(l.y));
    const unsigned long long num = f2fma(f2mul(f2dup(-k.a1), hf), slope, qn);
    const float2 den = f2unpack(f2fma(cq, r7, f2dup(1.0f)));
    const float2 v = f2unpack(f2mul(num, f2pack(rcp_fast(den.x), rcp_fast(den.y))));
    return f2pack(h.x > k.h_dry ? v.x : 0.0f, h.y > k.h_dry ? v.y : 0.0f);
}

// 16 bytes global -> shared, asynchronously (in the thread's current group); in == false: zeros.
__device__ __forceinline__ void copy16(float *dst, const float *src, bool in)
{
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"((unsigned)__cvta_generic_to_shared(dst)), "l"(src),
                 "r"(in ? 16 : 0)
                 : "memory");
}

__device__ __forceinline__ void copy_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }

template <int N>
__device__ __forceinline__ void copy_wait()
{
    asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory");
}

constexpr int kAhead = 2;                // rows in flight ahead of level 1 (a power of two)
constexpr int kRowsZ = 8;                // rows of z kept: those in flight, and back to the one below level K's
static_assert(kRowsZ >= kAhead + 4 + 1, "the z rows of four levels and those in flight");

// One warp's shared memory; every lane reads only what it copied or wrote itself.
template <int kMode>
struct alignas(16) TiledSmem {
    float raw[kAhead][3][128];           // level 1's rows in flight: h, qx, n
    float qy[kMode ? 4 : kAhead][128];   // and qy (the scheme options read it one row further on)
    float z[kRowsZ][128];
    float c[4][4][128];                  // face_c and the higher bed of a row's west and south faces, for levels 2 .. K
};

// One work item: strip `strip`, rows [y0, y1) of grid a, steps s0 .. s0 + K - 1 of the epoch.
//
// kMode bit 0: theta-weighted numerator discharges; bit 1: the vector norm in the friction term.
// A face then needs the old discharges around it: those of the row below are kept in registers
// (4 more per option and level), the old qy of the row above is the row that level s - 1 has just
// computed (level 1: the next row in flight).  A lane at the strip's edge takes its missing
// neighbour column as garbage, like the plain arithmetic's edge lanes: it stays inside the halo.
// kGauge: rows with gauges (a.gauge_row) go to a.gauge_rows after each of the K steps, the strip's own columns of them;
// one launch takes the gauges out after many steps.  So the kernel knows rows only, whatever the gauges' number and
// order.  (Recording from lists, every item testing all gauges, a crowded one scanning them at every tick, took
// 194 ms for 64 steps of 1024^2 with 4096 gauges in a 64 x 64 patch, 0.60 so, and 0.56 with one gauge, 0.55 so.)
template <int K, int kMode, bool kGauge>
__device__ __forceinline__ void tiled_item(const StepArgs<float> &a, const int s0, const int strip, const int y0,
                                           const int y1, const int want_hmax, TiledSmem<kMode> &sm)
{
    constexpr bool kTheta = (kMode & 1) != 0, kVec = (kMode & 2) != 0;
    constexpr int kOut = out_cols(K, kMode), kRowsQy = kMode ? 4 : kAhead;
    const Geom &G = a.geo;
    const int lane = threadIdx.x;
    const int nx = G.nx, ny = G.ny;
    const size_t P = (size_t)G.pitch;
    FastConst Kc;
    {
        const float dt = (float)a.ctrl->dt, dx = (float)G.dx, g = (float)G.g;
        Kc.gdt = g * dt;
        Kc.a1 = Kc.gdt / dx;
        Kc.gdt4 = 0.25f * Kc.gdt;
        Kc.h_dry = (float)G.h_dry;
        Kc.dtdx = dt / dx;
        Kc.theta = (float)G.theta;
        Kc.w = (float)(0.5 * (1.0 - G.theta));
    }
    const int x0 = strip * kOut - halo_cols(K);
    const int c0 = x0 + 4 * lane;
    const int own_lo = strip * kOut, own_hi = min(own_lo + kOut, nx);
    const bool west = x0 < 0, east = x0 + 127 >= nx;   // the strip holds a border column of the grid
    const bool in = c0 >= 0 && c0 < (int)P;            // the lane's columns lie in the rows (the pitch is a multiple of 4)
    const int jb = max(y0 - K, 0);
    const int jhi = min(y1 + K - 1, ny - 1);           // last staged row
    const int jlast = min(y1, ny) + K - 1;             // last tick: level K reaches row y1
    // Ticks at which every level's row lies inside the grid (rows 0 and ny have border faces): all levels
    // run, on garbage until their first rows arrive, which no row of the item depends on.
    const int steady_lo = jb > 0 ? jb : K, steady_hi = jhi;
    // lanes whose four columns the strip owns, and the one that owns some of them or only face nx
    const bool full = c0 >= own_lo && c0 + 3 < own_hi;
    const bool part = !full && c0 >= own_lo && (c0 < own_hi || (c0 == nx && own_hi == nx));
    const size_t lane_off = in ? (size_t)c0 : 0;

    auto issue = [&](int j) {
        if (j <= jhi) {
            const size_t o = (size_t)j * P + lane_off;
            float *d = &sm.raw[j & (kAhead - 1)][0][4 * lane];
            copy16(d, a.h + o, in);
            copy16(d + 128, a.qx + o, in);
            copy16(d + 256, a.n + o, in);
            copy16(&sm.z[j & (kRowsZ - 1)][4 * lane], a.z + o, in);
            if constexpr (kMode)                       // qy has a row more than the cells
                copy16(&sm.qy[(j + 1) & (kRowsQy - 1)][4 * lane], a.qy + o + P, in);
            else
                copy16(&sm.qy[j & (kRowsQy - 1)][4 * lane], a.qy + o, in);
        }
        copy_commit();                                 // a group per tick, empty past the last row
    };
    if constexpr (kMode) copy16(&sm.qy[jb & (kRowsQy - 1)][4 * lane], a.qy + (size_t)jb * P + lane_off, in);
    for (int j = jb; j < jb + kAhead; j++) issue(j);

    // The border faces at x = 0 and x = nx (Eq. 5-6): at the end of a tick lane s - 1 evaluates level s's
    // west one and lane 4 + s - 1 its east one, side by side, and hands them to the lanes that hold them
    // (each level for itself, in line, cost 600 cycles a level).  Type, inflow slot, sqrt(S) and n of the
    // cell are read a tick ahead.
    const int bl = lane & 3, bs = (lane >> 2) & 1;     // this lane's level - 1 and side
    const bool border = lane < 8 && bl < K && (bs ? east : west);
    const int cell_lane = (nx - 1 - x0) >> 2, cell_k = (nx - 1) & 3;   // where column nx - 1 lies (if east)
    const int face_lane = (nx - x0) >> 2, face_k = nx & 3;             // where face nx lies
    int nb_t = kBcWall, nb_s = 0;
    float nb_q = 0.0f, nb_n = 1.0f;
    auto border_fetch = [&](int r) {
        nb_t = kBcWall;
        if (border && r >= jb && r <= jhi) {
            const int off = (bs ? ny : 0) + r;
            nb_t = a.bc.type[off];
            nb_s = a.bc.slot[off];
            nb_q = a.bc.sqrtS_f[off];
            nb_n = a.n[(size_t)r * P + (bs ? nx - 1 : 0)];
        }
    };
    border_fetch(jb - bl);

    unsigned gm = 0;                                   // (kGauge) bit s - 1 at tick j: row j - s has a place
    const bool keep = c0 >= own_lo && c0 < own_hi;     // (a lane with the grid's last columns stores some padding too)
    auto gauge_store = [&](int s, int r, const Row4 &v) {
        if (((gm >> (s - 1)) & 1) && keep)
            row_store(a.gauge_rows + ((size_t)(s - 1) * a.n_gauges + __ldg(a.gauge_row + r)) * P + lane_off, v);
    };

    Row4 sh[K], sx[K], sy[K];                          // per level: the previous row's old depth and new faces
    Row4 ox[K], oy[K];                                 // the sums of its neighbouring old qx (kVec), its old qy (kTheta)
    Row4 pn{0, 0};                                     // n of the previous row (level 1)
#pragma unroll
    for (int s = 0; s < K; s++) sh[s] = sx[s] = sy[s] = ox[s] = oy[s] = Row4{0, 0};
    float fq = 0.0f, fc = 0.0f;                        // boundary outflow and clipped depth since the last fold
    double led_q = 0.0, led_c = 0.0;
    float hmax = 0.0f;

    auto tick = [&](auto steady_t, auto edge_t, const int j) {
        constexpr bool kSteady = decltype(steady_t)::value, kEdge = decltype(edge_t)::value;
        Row4 ch{0, 0}, cx{0, 0}, cy{0, 0}, cyn{0, 0};  // the current level's input row, and the old qy of the row above it
        int place = -1;                                // of row j
        if (kGauge && j >= y0 && j < y1) place = __ldg(a.gauge_row + j);
        copy_wait<kAhead - 1>();
#pragma unroll
        for (int s = 1; s <= K; s++) {
            const int r = j - (s - 1);
            const int rstart = jb == 0 ? 0 : jb + (s - 1);
            if (kSteady || (r >= rstart && r <= ny && r <= y1 + K - s)) {
                const bool row = kSteady || r < ny;    // r == ny: only the north border faces
                Row4 z{0, 0}, pz{0, 0}, fcx{0, 0}, fcy{0, 0}, zx{0, 0}, zy{0, 0};
                if (row) z = row_load(&sm.z[r & (kRowsZ - 1)][4 * lane]);
                if (kSteady || r > 0) pz = row_load(&sm.z[(r - 1) & (kRowsZ - 1)][4 * lane]);
                if (s == 1) {
                    if (row) {
                        const float *d = &sm.raw[r & (kAhead - 1)][0][4 * lane];
                        ch = row_load(d);
                        cx = row_load(d + 128);
                        cy = row_load(&sm.qy[r & (kRowsQy - 1)][4 * lane]);
                        if constexpr (kMode) cyn = row_load(&sm.qy[(r + 1) & (kRowsQy - 1)][4 * lane]);
                        const Row4 n = row_load(d + 256);
                        const float2 n0 = f2unpack(n.a), n1 = f2unpack(n.b);
                        const float nl = from_left(n);
                        fcx.a = face_c(f2pack(__fadd_rn(nl, n0.x), __fadd_rn(n0.x, n0.y)), Kc);
                        fcx.b = face_c(f2pack(__fadd_rn(n0.y, n1.x), __fadd_rn(n1.x, n1.y)), Kc);
                        fcy.a = face_c(f2add(pn.a, n.a), Kc);
                        fcy.b = face_c(f2add(pn.b, n.b), Kc);
                        pn = n;
                        const Row4 zl = row_left(z, from_left(z));
                        zx = Row4{f2max(zl.a, z.a), f2max(zl.b, z.b)};
                        zy = Row4{f2max(pz.a, z.a), f2max(pz.b, z.b)};
                        if (K > 1) {
                            row_store(&sm.c[r & 3][0][4 * lane], fcx);
                            row_store(&sm.c[r & 3][1][4 * lane], fcy);
                            row_store(&sm.c[r & 3][2][4 * lane], zx);
                            row_store(&sm.c[r & 3][3][4 * lane], zy);
                        }
                    }
                    issue(j + kAhead);                 // into the slots just read
                } else if (row) {
                    fcx = row_load(&sm.c[r & 3][0][4 * lane]);
                    fcy = row_load(&sm.c[r & 3][1][4 * lane]);
                    zx = row_load(&sm.c[r & 3][2][4 * lane]);
                    zy = row_load(&sm.c[r & 3][3][4 * lane]);
                }
                if (!kSteady && r == rstart && jb > 0) {
                    sh[s - 1] = ch;                    // halo row: only becomes the previous row
                    if constexpr (kTheta) oy[s - 1] = cy;
                    if constexpr (kVec) {
                        const Row4 c1 = row_right(cx, from_right(cx));
                        ox[s - 1] = Row4{f2add(cx.a, c1.a), f2add(cx.b, c1.b)};
                    }
                } else {
                    Row4 &h0 = sh[s - 1], &x0r = sx[s - 1], &y0r = sy[s - 1];
                    const Row4 e{f2add(ch.a, z.a), f2add(ch.b, z.b)};
                    Row4 px{0, 0};                     // qx of the row's cells, west + east (kVec)
                    if constexpr (kVec) {
                        const Row4 c1 = row_right(cx, from_right(cx));
                        px = Row4{f2add(cx.a, c1.a), f2add(cx.b, c1.b)};
                    }
                    // ---- new south faces of row r
                    Row4 qs;
                    if (kSteady || (r > 0 && r < ny)) {
                        const Row4 ep{f2add(h0.a, pz.a), f2add(h0.b, pz.b)};
                        Row4 qn = cy, cq;
                        if constexpr (kTheta) {
                            qn.a = theta_q_x2(cy.a, oy[s - 1].a, cyn.a, Kc);
                            qn.b = theta_q_x2(cy.b, oy[s - 1].b, cyn.b, Kc);
                        }
                        if constexpr (kVec) {          // the mean of the old qx of rows r - 1 and r around the face
                            cq.a = f2mul(fcy.a, q_norm_sums_x2(cy.a, ox[s - 1].a, px.a));
                            cq.b = f2mul(fcy.b, q_norm_sums_x2(cy.b, ox[s - 1].b, px.b));
                        } else {
                            cq = Row4{face_cq(fcy.a, cy.a), face_cq(fcy.b, cy.b)};
                        }
                        qs.a = faces2(f2sub(f2max(ep.a, e.a), zy.a), f2sub(e.a, ep.a), qn.a, cq.a, Kc);
                        qs.b = faces2(f2sub(f2max(ep.b, e.b), zy.b), f2sub(e.b, ep.b), qn.b, cq.b, Kc);
                    } else {
                        // rows 0 and ny: Eq. 5-6
                        float v[4] = {0.0f, 0.0f, 0.0f, 0.0f};
                        const Row4 hb = r == 0 ? ch : h0;
                        const bool book = (r == 0 && y0 == 0) || (r == ny && y1 == ny);
#pragma unroll 1
                        for (int k = 0; k < 4; k++) {
                            const int c = c0 + k;
                            if (c < 0 || c >= nx) continue;
                            float qo = 0.0f;
                            const float h = k == 0 ? row_get(hb, 0) : k == 1 ? row_get(hb, 1) : k == 2 ? row_get(hb, 2) : row_get(hb, 3);
                            const float w = boundary_fast_flux(a, s0 + s - 1, r == 0 ? 2 : 3, c, h,
                                                               a.n[(size_t)(r == 0 ? 0 : ny - 1) * P + c], qo);
                            if (book && c >= own_lo && c < own_hi) fq += qo;
                            if (k == 0) v[0] = w;
                            else if (k == 1) v[1] = w;
                            else if (k == 2) v[2] = w;
                            else v[3] = w;
                        }
                        qs = row_pack(v[0], v[1], v[2], v[3]);
                    }
                    // ---- finish row r-1: Eq. 4 and the clip
                    Row4 fin{0, 0};
                    const bool has_prev = kSteady || (jb == 0 ? r > 0 : r > rstart + 1);
                    if (has_prev) {
                        const int rr = r - 1;
                        const float2 x01 = f2unpack(x0r.a), x23 = f2unpack(x0r.b);
                        const float xe = from_right(x0r);
                        const unsigned long long dx0 = f2pack(__fsub_rn(x01.x, x01.y), __fsub_rn(x01.y, x23.x));
                        const unsigned long long dx1 = f2pack(__fsub_rn(x23.x, x23.y), __fsub_rn(x23.y, xe));
                        fin.a = f2fma(f2dup(Kc.dtdx), f2add(dx0, f2sub(y0r.a, qs.a)), h0.a);
                        fin.b = f2fma(f2dup(Kc.dtdx), f2add(dx1, f2sub(y0r.b, qs.b)), h0.b);
                        const float2 f0 = f2unpack(fin.a), f1 = f2unpack(fin.b);
                        if ((__float_as_int(f0.x) | __float_as_int(f0.y) | __float_as_int(f1.x) | __float_as_int(f1.y)) < 0) {   // a sign bit (rare): clip, book the removed volume
                            const bool book = rr >= y0 && rr < y1 && rr >= G.led_j0 && rr < G.led_j1;
                            float v[4] = {f0.x, f0.y, f1.x, f1.y};
#pragma unroll
                            for (int k = 0; k < 4; k++)
                                if (v[k] < 0.0f) {
                                    if (book && c0 + k >= own_lo && c0 + k < own_hi) fc -= v[k];
                                    v[k] = 0.0f;
                                }
                            fin = row_pack(v[0], v[1], v[2], v[3]);
                        }
                        if (s == K && rr >= y0 && (kSteady || rr < y1)) {
                            const float2 g0 = f2unpack(fin.a), g1 = f2unpack(fin.b);
                            const size_t ro = (size_t)rr * P + lane_off;
                            const bool north = !kSteady && rr == ny - 1;   // the grid's north face row too
                            if (kGauge) gauge_store(K, rr, fin);
                            const bool maximum = want_hmax && rr >= G.led_j0 && rr < G.led_j1;   // a part's own rows
                            if (kEdge ? full : lane >= 1 && lane <= kOut / 4) {
                                if (maximum) hmax = max_nan(max_nan(hmax, max_nan(g0.x, g0.y)), max_nan(g1.x, g1.y));
                                row_store(a.h_out + ro, fin);
                                row_store(a.qx_out + ro, x0r);
                                row_store(a.qy_out + ro, y0r);
                                if (north) row_store(a.qy_out + ro + P, qs);
                            } else if (kEdge && part) {
                                const float f[4] = {g0.x, g0.y, g1.x, g1.y};
#pragma unroll
                                for (int k = 0; k < 4; k++) {
                                    const int c = c0 + k;
                                    if (c < own_hi) {
                                        if (maximum) hmax = max_nan(hmax, f[k]);
                                        a.h_out[ro + k] = f[k];
                                        a.qy_out[ro + k] = row_get(y0r, k);
                                        if (north) a.qy_out[ro + P + k] = row_get(qs, k);
                                    }
                                    if (c < own_hi || c == nx) a.qx_out[ro + k] = row_get(x0r, k);
                                }
                            }
                        }
                    }
                    // ---- new west faces of row r; it becomes this level's previous row, and the
                    // finished one the next level's input
                    Row4 qx{0, 0};
                    if (row) {
                        const Row4 el = row_left(e, from_left(e));
                        Row4 qn = cx, cq;
                        if constexpr (kTheta) {
                            const Row4 l = row_left(cx, from_left(cx)), n = row_right(cx, from_right(cx));
                            qn.a = theta_q_x2(cx.a, l.a, n.a, Kc);
                            qn.b = theta_q_x2(cx.b, l.b, n.b, Kc);
                        }
                        if constexpr (kVec) {          // the mean of the old qy of rows r and r + 1 around the face
                            const Row4 yl = row_left(cy, from_left(cy)), nl = row_left(cyn, from_left(cyn));
                            cq.a = f2mul(fcx.a, q_norm_x2(cx.a, yl.a, cy.a, nl.a, cyn.a));
                            cq.b = f2mul(fcx.b, q_norm_x2(cx.b, yl.b, cy.b, nl.b, cyn.b));
                        } else {
                            cq = Row4{face_cq(fcx.a, cx.a), face_cq(fcx.b, cx.b)};
                        }
                        // (the slopes scalar: the packed form would copy the shifted pairs together first)
                        const float2 e0 = f2unpack(e.a), e1 = f2unpack(e.b), l0 = f2unpack(el.a);
                        const unsigned long long s0_ = f2pack(__fsub_rn(e0.x, l0.x), __fsub_rn(e0.y, e0.x));
                        const unsigned long long s1_ = f2pack(__fsub_rn(e1.x, e0.y), __fsub_rn(e1.y, e1.x));
                        qx.a = faces2(f2sub(f2max(el.a, e.a), zx.a), s0_, qn.a, cq.a, Kc);
                        qx.b = faces2(f2sub(f2max(el.b, e.b), zx.b), s1_, qn.b, cq.b, Kc);
                    }
                    const Row4 hx = x0r, hy = y0r;
                    h0 = ch;
                    if constexpr (kTheta) oy[s - 1] = cy;
                    if constexpr (kVec) ox[s - 1] = px;
                    x0r = qx;
                    y0r = qs;
                    ch = fin;
                    cx = hx;
                    cy = hy;
                    if constexpr (kMode) cyn = qs;     // the next level's row lies below this level's row r
                }
            } else if (s == 1) {
                issue(j + kAhead);
            }
        }
        if constexpr (kGauge) {
            // level s finished row j - s, the next level's previous row (level K stored its own above)
            if (gm & ((1u << (K - 1)) - 1)) {
#pragma unroll
                for (int s = 1; s < K; s++) gauge_store(s, j - s, sh[s]);
            }
            gm = gm << 1 | (place >= 0 ? 1u : 0u);
        }
        if (kEdge && (west || east)) {
            float h = 0.0f;
#pragma unroll
            for (int s = 0; s < K; s++) {
                if (west) {
                    const float v = __shfl_sync(0xffffffffu, f2unpack(sh[s].a).x, halo_cols(K) / 4);
                    if (lane == s) h = v;
                }
                if (east) {
                    const float2 p = f2unpack(cell_k < 2 ? sh[s].a : sh[s].b);
                    const float v = __shfl_sync(0xffffffffu, (cell_k & 1) ? p.y : p.x, cell_lane);
                    if (lane == 4 + s) h = v;
                }
            }
            float f = 0.0f;
            if (nb_t != kBcWall) {
                const int r = j - bl;
                if (nb_t == kBcInflow) {
                    f = a.inflow_q[(size_t)(s0 + bl) * a.n_slots + nb_s];
                } else {
                    f = outflow_fast(h, nb_q, nb_n, G.dx_f, G.h_dry_f, G.bc_form);
                    if (nb_t == kBcOutflow && r >= y0 && r < y1 && (bs ? own_hi == nx : own_lo == 0)) fq += f;
                    f = -f;
                }
                if (bs) f = -f;
            }
            border_fetch(j + 1 - bl);
#pragma unroll
            for (int s = 0; s < K; s++) {
                if (west) {
                    const float v = __shfl_sync(0xffffffffu, f, s);
                    const float2 p = f2unpack(sx[s].a);
                    sx[s].a = f2pack(lane == halo_cols(K) / 4 ? v : p.x, p.y);
                }
                if (east) {
                    const float v = __shfl_sync(0xffffffffu, f, 4 + s);
                    const bool mine = lane == face_lane;
                    const float2 p = f2unpack(sx[s].a), q = f2unpack(sx[s].b);
                    sx[s].a = f2pack(mine && face_k == 0 ? v : p.x, mine && face_k == 1 ? v : p.y);
                    sx[s].b = f2pack(mine && face_k == 2 ? v : q.x, mine && face_k == 3 ? v : q.y);
                }
            }
        }
    };

    int j = jb;
    while (j <= jlast) {
        // runs of at most 32 ticks, after which the float partial sums are folded into double ones
        const int jend = min(j + 31, jlast);
        if (j >= steady_lo && j <= steady_hi) {
            const int e = min(jend, steady_hi);
            if (west || east) {
#pragma unroll 1
                for (; j <= e; j++) tick(std::true_type{}, std::true_type{}, j);
            } else {
#pragma unroll 1
                for (; j <= e; j++) tick(std::true_type{}, std::false_type{}, j);
            }
        } else {
            const int e = j < steady_lo ? min(jend, steady_lo - 1) : jend;
#pragma unroll 1
            for (; j <= e; j++) tick(std::false_type{}, std::true_type{}, j);
        }
        if (__any_sync(0xffffffffu, fq != 0.0f || fc != 0.0f)) {   // rare: boundary faces, clipped cells
            led_q += warp_sum((double)fq);
            led_c += warp_sum((double)fc);
            fq = fc = 0.0f;
        }
    }
    copy_wait<0>();
    if (lane == 0) {
        if (led_q != 0.0) atomicAdd(&a.ctrl->V_out, a.ctrl->dt * led_q * G.dx);
        if (led_c != 0.0) atomicAdd(&a.ctrl->V_clip, led_c * G.dx * G.dx);
    }
    if (want_hmax) {
        for (int o = 16; o > 0; o >>= 1) hmax = max_nan(hmax, __shfl_xor_sync(0xffffffffu, hmax, o));
        if (lane == 0) atomic_max_nonneg(&a.ctrl->hmax_bits, hmax != hmax ? (double)NAN : (double)hmax);
    }
}

// Inflow volume of the K steps and the clock after them (one thread per grid).
template <int K>
__device__ __forceinline__ void tiled_finish(const StepArgs<float> &a, const int s0)
{
    const double dtd = a.ctrl->dt;
    double vin = a.ctrl->V_in;
    for (int s = 0; s < K; s++)
        for (int k = 0; k < a.n_inflow_sec; k++) {
            const double Q = a.inflow_Q[(size_t)(s0 + s) * a.n_inflow_sec + k];
            if (Q > 0.0) vin += dtd * Q;
        }
    a.ctrl->V_in = vin;
    a.ctrl->t = a.t_list[s0 + K];
}

// Item `item` of grid a (a.tile_y rows per item, a.tile_x in the edge strips).
template <int K, int kMode, bool kGauge>
__device__ __forceinline__ void tiled_run(const StepArgs<float> &a, const int s0, const int item, const int want_hmax,
                                          TiledSmem<kMode> &sm)
{
    constexpr int kOut = out_cols(K, kMode);
    const int n_strips = (a.geo.nx + kOut - 1) / kOut, n_edge = min(n_strips, 2);
    const int edge_items = n_edge * ((a.geo.ny + a.tile_x - 1) / a.tile_x);
    int strip, y0, rows;
    if (item < edge_items) {
        strip = item % n_edge ? n_strips - 1 : 0;
        rows = a.tile_x;
        y0 = (item / n_edge) * rows;
    } else {
        strip = 1 + (item - edge_items) % (n_strips - n_edge);
        rows = a.tile_y;
        y0 = (item - edge_items) / (n_strips - n_edge) * rows;
    }
    tiled_item<K, kMode, kGauge>(a, s0, strip, y0, min(y0 + rows, a.geo.ny), want_hmax, sm);
}

// One grid: a block per item, or (a caller's cap on the pipelines) gridDim.x blocks that walk the items.
template <int K, int kMode, bool kGauge>
__global__ void __launch_bounds__(32, tiled_warps(kMode)) step_tiled_kernel(const __grid_constant__ StepArgs<float> a)
{
    __shared__ TiledSmem<kMode> sm;
    pdl_wait();
    pdl_launch();
    const int n_items = tiled_item_count(a.geo.nx, a.geo.ny, out_cols(K, kMode), a.tile_y, a.tile_x);
#pragma unroll 1
    for (int item = blockIdx.x; item < n_items; item += gridDim.x) tiled_run<K, kMode, kGauge>(a, a.s, item, a.want_hmax, sm);
    if (blockIdx.x == 0 && threadIdx.x == 0) tiled_finish<K>(a, a.s);
}

// The grid whose items base[k] .. base[k+1] - 1 hold `item`.
__device__ __forceinline__ int grid_of_item(const int *base, const int n, const int item)
{
    int lo = 0, hi = n - 1;
    while (lo < hi) {
        const int mid = (lo + hi + 1) >> 1;
        if (base[mid] <= item) lo = mid;
        else hi = mid - 1;
    }
    return lo;
}

// An item of one of many grids.  The grid's first item books its inflow volume and clock.  (The items are
// numbered for the table's K; a shorter launch's strips may be wider.)
template <int K, int kMode>
__device__ __forceinline__ void tiled_run_of_many(const StepArgs<float> &a, const int s0, const int local, const int want_hmax,
                                                  TiledSmem<kMode> &sm)
{
    if (local == 0 && threadIdx.x == 0) tiled_finish<K>(a, s0);
    if (local >= tiled_item_count(a.geo.nx, a.geo.ny, out_cols(K, kMode), a.tile_y, a.tile_x)) return;
    tiled_run<K, kMode, false>(a, s0, local, want_hmax, sm);
}

// Many grids: the items of grid k (table[k].tile_x and tile_y rows per item) are numbered
// base[k] .. base[k+1] - 1, grids ordered largest first; a block per item.  With the grids' arguments in
// the launch's own (step_tiled_grids_kernel) they are read from constant memory as a single grid's are;
// more than fit there come from a table on the device, and the block keeps its grid's in shared memory
// (12 more registers, and an item starts with two round trips to memory).  One strip of 16384^2 / 4096^2, us a step: 473 / 40.4
// and 508 / 43.0 (the single grid's kernel 463 / 39.1).
template <int N>
struct GridArgs {
    StepArgs<float> grid[N];
    int base[N + 1];
};
constexpr int kFewGrids = 12, kManyGrids = 104;    // arguments of 4 and 32 KB, the sizes a launch may have
static_assert(sizeof(GridArgs<kFewGrids>) + 16 <= 4096 && sizeof(GridArgs<kManyGrids>) + 16 <= 32764, "kernel arguments");

template <int K, int kMode, int N>
__global__ void __launch_bounds__(32, tiled_warps(kMode))
    step_tiled_grids_kernel(const __grid_constant__ GridArgs<N> g, const int n, const int s0, const int want_hmax)
{
    __shared__ TiledSmem<kMode> sm;
    const int k = grid_of_item(g.base, n, blockIdx.x);
    tiled_run_of_many<K, kMode>(g.grid[k], s0, (int)blockIdx.x - g.base[k], want_hmax, sm);
}

template <int K, int kMode>
__global__ void __launch_bounds__(32, tiled_warps(kMode))
    step_tiled_ensemble_kernel(const StepArgs<float> *table, const int *base, const int n, const int s0, const int want_hmax)
{
    __shared__ TiledSmem<kMode> sm;
    __shared__ StepArgs<float> a;
    const int item = blockIdx.x, lo = grid_of_item(base, n, item);
    static_assert(sizeof(StepArgs<float>) % 8 == 0, "copied in 8-byte words");
    for (int w = threadIdx.x; w < (int)(sizeof(StepArgs<float>) / 8); w += 32)
        reinterpret_cast<unsigned long long *>(&a)[w] = reinterpret_cast<const unsigned long long *>(table + lo)[w];
    __syncwarp();
    tiled_run_of_many<K, kMode>(a, s0, item - base[lo], want_hmax, sm);
}

template <int K, int kMode>
cudaError_t launch_k(const StepArgs<float> &a0, cudaStream_t st)
{
    StepArgs<float> a = a0;
    const int nx = a.geo.nx, ny = a.geo.ny, out = out_cols(K, kMode);
    int rows = 0, edge = 0, blocks = 0;
    if (a0.tile_y > 0) rows = edge = a0.tile_y < ny ? a0.tile_y : ny;   // caller's rows per work item
    else if (a0.tile_x > 0) {
        tiled_split_dynamic((nx + out - 1) / out, ny, a0.tile_x, K, &rows, &blocks);
        edge = rows;
    } else tiled_rows(nx, ny, K, kMode, &rows, &edge);
    const int items = tiled_item_count(nx, ny, out, rows, edge);
    blocks = a0.tile_x > 0 && a0.tile_x < items ? a0.tile_x : items;    // caller's cap on pipelines
    a.tile_x = edge;
    a.tile_y = rows;
    return launch_pdl(a.gauge_rows ? step_tiled_kernel<K, kMode, true> : step_tiled_kernel<K, kMode, false>,
                      blocks, 32, st, a);
}

// Launchers of one scheme mode for every steps-per-launch K.
template <int kMode>
cudaError_t launch_tiled_mode(const StepArgs<float> &a, cudaStream_t st)
{
    switch (a.k_steps) {
    case 1: return launch_k<1, kMode>(a, st);
    case 2: return launch_k<2, kMode>(a, st);
    case 3: return launch_k<3, kMode>(a, st);
    case 4: return launch_k<4, kMode>(a, st);
    default: return cudaErrorInvalidValue;
    }
}

template <int K, int kMode, int N>
cudaError_t launch_grids(const GridTable &t, int s0, int want_hmax, cudaStream_t st)
{
    GridArgs<N> g = {};
    for (int k = 0; k < t.n; k++) g.grid[k] = t.host_table[k];
    for (int k = 0; k <= t.n; k++) g.base[k] = t.host_base[k];
    step_tiled_grids_kernel<K, kMode, N><<<t.host_base[t.n], 32, 0, st>>>(g, t.n, s0, want_hmax);
    return cudaGetLastError();
}

// (The arguments' form is built for K = 4, the steps of nearly every launch.)
template <int kMode>
cudaError_t launch_tiled_ensemble_mode(const GridTable &t, int k_steps, int s0, int want_hmax, cudaStream_t st)
{
    const int items = t.host_base[t.n];
    if (items < 1) return cudaSuccess;
    if (k_steps == 4 && t.n <= kFewGrids) return launch_grids<4, kMode, kFewGrids>(t, s0, want_hmax, st);
    if (k_steps == 4 && t.n <= kManyGrids) return launch_grids<4, kMode, kManyGrids>(t, s0, want_hmax, st);
    switch (k_steps) {
    case 1: step_tiled_ensemble_kernel<1, kMode><<<items, 32, 0, st>>>(t.table, t.base, t.n, s0, want_hmax); break;
    case 2: step_tiled_ensemble_kernel<2, kMode><<<items, 32, 0, st>>>(t.table, t.base, t.n, s0, want_hmax); break;
    case 3: step_tiled_ensemble_kernel<3, kMode><<<items, 32, 0, st>>>(t.table, t.base, t.n, s0, want_hmax); break;
    case 4: step_tiled_ensemble_kernel<4, kMode><<<items, 32, 0, st>>>(t.table, t.base, t.n, s0, want_hmax); break;
    default: return cudaErrorInvalidValue;
    }
    return cudaGetLastError();
}

}  // namespace

}  // namespace flood
