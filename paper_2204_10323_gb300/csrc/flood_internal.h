// flood_internal.h -- plain structs shared by the runtime (flood_api.cpp) and
// the CUDA kernels.  No PyTorch types; included by host C++ and by nvcc.
#pragma once

#include <cstddef>
#include <cstdint>
#include <cuda_runtime.h>

namespace flood {

constexpr int kMaxEpoch = 1024;       // largest E (steps per CFL epoch)
constexpr int kBcWall = 0, kBcInflow = 1, kBcOutflow = 2;
// An outflow face of a subdomain's halo row: its flux is computed like any
// outflow face but its volume is booked by the subdomain that owns the row.
constexpr int kBcOutflowHalo = 3;

// Device status bits (sticky, OR-ed by kernels).
constexpr int kStatusNonfinite = 1;
constexpr int kStatusTimeout = 2;
constexpr int kStatusCfl = 4;          // an epoch's dt broke the Courant limit dx / sqrt(g h_max) at its end

// Device-resident control block of one simulation.
struct Ctrl {
    double t;                     // time at the start of the next step
    double dt;                    // time step of the current epoch
    double V_in, V_out, V_clip;   // cumulative volumes (m^3)
    double h_max;                 // depth maximum measured at the current epoch start
    double cfl_exceed;            // epochs whose dt broke dx / sqrt(g h_max) at their end
    unsigned long long hmax_bits; // running max of h (bits of a non-negative double)
    int status;                   // kStatus* bits
    unsigned epoch_blocks;        // blocks of an epoch start that have read the words above (0 between epoch starts)
};

// One inflow section as seen by the Eq. 6 solver.
struct InflowSec {
    int ncell;                    // cells along the section
    int cell0;                    // offset into the section cell-index array
    int slot0;                    // first column of this section in the per-step flux rows
    int tab0, ntab;               // hydrograph table offset / length
    int side;                     // flood_side of the section
    double sqrtS;                 // sqrt(S_in)
};

// Geometry and physical constants (both precisions keep them in double here;
// kernels cast to their working type).
struct Geom {
    int nx, ny;
    int pitch;                    // elements per row of every grid array
    int bc_form;
    double dx, g, h_dry;
    float dx_f, h_dry_f;          // dx and h_dry rounded to FP32 once (the fast kernels' boundary faces)
    double theta;                 // face-flux weighting (1 = Eq. 3 as printed)
    int friction;                 // |q| of the friction term: 0 the face's own, 1 the vector norm
    double cfl_alpha, dt_cap, dt_const;
    int dt_mode, epoch_steps;
    int led_j0, led_j1;           // rows whose clipped volume and stored volume this grid books (all rows,
                                  // except for a subdomain of a decomposed grid: its own rows)
};

// Boundary description, one entry per boundary cell: sides laid out as
// [xmin: ny][xmax: ny][ymin: nx][ymax: nx].
struct Boundary {
    const int8_t *type;           // kBcWall / kBcInflow / kBcOutflow
    const int32_t *slot;          // inflow: column in the per-step inflow flux row
    const double *sqrtS;          // outflow: sqrt(S_out)
    const float *sqrtS_f;         // the same rounded to FP32 (fast kernels)
};

template <typename T>
struct StepArgs {
    Geom geo;
    const T *h, *qx, *qy, *z, *n;
    T *h_out, *qx_out, *qy_out;
    Boundary bc;
    const T *inflow_q;            // E x n_slots unit-width inflow fluxes (into the domain)
    int n_slots;
    const double *inflow_Q;       // E x n_inflow_sections discharges (for V_in)
    int n_inflow_sec;
    const double *t_list;         // E + 1 start times of the epoch's steps
    Ctrl *ctrl;
    int s;                        // step index inside the epoch (first step of the launch)
    int k_steps;                  // steps done by this launch (1 except the tiled kernel)
    int want_hmax;                // 1: record max depth after the launch's last step
    // Gauges after every step: n_gauges cells (flat j*nx+i) into n_gauges values of gauge_out (null: none).  Tiled:
    // whole rows of depths instead, row r into place gauge_row[r] (< 0: none) of the step's n_gauges rows of `pitch`
    // floats in gauge_rows (k_steps x n_gauges rows; null: none).
    union {
        const int64_t *gauge_cells;
        const int *gauge_row;
    };
    int n_gauges;
    union {
        double *gauge_out;
        float *gauge_rows;
    };
    int tile_x, tile_y;           // launch shape (stream/TMA: warps, rows; tiled: rows per item of the edge
                                  // strips and of the others; on its way in: cap on pipelines, rows per item)
};

// ---------------------------------------------------------------- launchers
// Each returns the cudaError_t of the launch.
template <typename T>
cudaError_t launch_step_reference(const StepArgs<T> &a, cudaStream_t st);
cudaError_t launch_step_rows(const StepArgs<float> &a, cudaStream_t st);
cudaError_t launch_step_stream(const StepArgs<float> &a, cudaStream_t st);
// Stream kernel over many grids: table of per-grid arguments (device), block
// prefix base[n+1] (device), one launch of total_blocks blocks.
// mode: the scheme options shared by every grid (bit 0 theta weighting, bit 1 vector-norm friction).
cudaError_t launch_step_stream_ensemble(const StepArgs<float> *table, const int *base, int n, int total_blocks,
                                        int warps, int rows, int step, int want_hmax, int mode, cudaStream_t st);
// Blocks of one grid for the stream kernel, and the (warps, rows) a tile pair selects.
int stream_blocks(const Geom &g, int warps, int rows);
cudaError_t launch_step_tma(const StepArgs<float> &a, cudaStream_t st);
// Temporal blocking over many grids, k_steps steps from s0: the items of grid k are base[k] .. base[k+1] - 1
// (tiled_items per grid, table[k].tile_y rows per item, tile_x in the edge strips).
int tiled_items(const Geom &g, int rows, int rows_edge, int k_steps);
// Multiprocessors of the GPU (152 where there is none), and the one-warp items of a scheme mode that it holds at once.
int sm_count();
int tiled_resident(int mode);
// Rows per work item (inner strips, and the one or two strips with the borders x = 0 and x = nx) for a grid
// alone on the GPU.
void tiled_rows(int nx, int ny, int K, int mode, int *rows, int *rows_edge);
void tiled_rows_for(int n_strips, int ny, int repeat, int warps, double base, double slope, double edge_more, int *rows,
                    int *rows_edge);
struct GridTable {
    const StepArgs<float> *table, *host_table;    // n grids: on the device, and the same on the host
    const int *base, *host_base;                  // n + 1
    int n;
};
cudaError_t launch_step_tiled_ensemble(const GridTable &t, int k_steps, int s0, int want_hmax, int mode, cudaStream_t st);
void stream_launch_shape(const Geom &g, int tile_x, int tile_y, int *warps, int *rows);
cudaError_t launch_step_tiled(const StepArgs<float> &a, cudaStream_t st);

// Decomposed grid: every part's running h_max (ctrls: n device pointers, on
// the device) set to the largest of them.
cudaError_t launch_hmax_allreduce(Ctrl *const *ctrls, int n, cudaStream_t st);
// What an epoch start of one simulation reads and writes.
template <typename T>
struct EpochArgs {
    Geom geo;
    Ctrl *ctrl;
    double *t_list;
    const InflowSec *secs;
    int nsec;
    const int64_t *cells;
    const double *tab_t, *tab_q;
    const T *z, *n;
    T *inflow_q;
    int n_slots;
    double *inflow_Q, *inflow_W;
};
// Eq. 6 for every (step of the epoch, inflow section) pair.  begin: the epoch starts: choose dt from h_max (or
// constant, or fixed_dt[0] when given: the adjoint's replay of a logged epoch), fill t_list, reset the running
// maximum, count CFL exceedances, flag NaN/Inf; else Eq. 6 alone, from the t_list there is.
template <typename T>
cudaError_t launch_inflow(const EpochArgs<T> &A, int E, bool begin, const double *fixed_dt, cudaStream_t st);
// Epoch starts of a batch of simulations (task = {simulation, section}); all_inflow: every one has a section
// (one launch, else two).
template <typename T>
cudaError_t launch_epoch_batched(const EpochArgs<T> *tab, int n, const int2 *tasks, int n_tasks, int E, bool all_inflow,
                                 cudaStream_t st);
// h_max of a state into ctrl->hmax_bits (max with what is there).
template <typename T>
cudaError_t launch_hmax(const Geom &g, const T *h, Ctrl *ctrl, cudaStream_t st);
// rows of `width` bytes from src to dst (device memory of the current device), pitches in bytes.
cudaError_t launch_copy_rows(void *dst, size_t dpitch, const void *src, size_t spitch, size_t width, size_t rows,
                             cudaStream_t st);
// n copies of `units` 16-byte units each (device memory, 16-byte aligned), max_units the longest.
struct HaloRows {
    const void *src;
    void *dst;
    int64_t units;
};
cudaError_t launch_halo_rows(const HaloRows *copies, int n, int64_t max_units, cudaStream_t st);
// Block mean (f x f, partial blocks at the far edges) of a ny x nx field into ceil(ny/f) x ceil(nx/f).
template <typename T>
cudaError_t launch_coarsen(const T *src, int nx, int ny, int f, T *dst, cudaStream_t st);
// OR of "some element is NaN or Inf" over rows x cols of a pitched array into *flag (device).
template <typename T>
cudaError_t launch_nonfinite(const T *a, int rows, int cols, int pitch, int *flag, cudaStream_t st);
// Deterministic two-pass sum of h * dx^2 into *out (double, device).
template <typename T>
cudaError_t launch_volume(const Geom &g, const T *h, double *partials, int n_partials, double *out,
                          cudaStream_t st);
// ---------------------------------------------------------------- adjoint
// Buffers of one reverse step (all pitched like the state; gn in double).
template <typename T>
struct AdjArgs {
    StepArgs<T> fwd;              // forward state x_k (h, qx, qy, z, n), BCs, inflow row, ctrl (dt)
    const T *lh, *lqx, *lqy;      // adjoint of x_{k+1}
    T *lh_out, *lqx_out, *lqy_out;   // adjoint of x_k
    T *lhu;                       // scratch: adjoint of the unclipped depth
    double *gn;                   // dL/dn accumulator
    const InflowSec *secs;        // inflow sections (for the Eq. 6 derivative)
    const int64_t *sec_cells;
    const double *inflow_W;       // E x n_sec levels of this epoch
    const int64_t *gauge_cells;   // flat j*nx+i of the loss's gauges
    const int4 *gauge_list;       // FP32, Eq. 3 as printed: the same as (row, column, index), in that order
    int n_gauges;
    const double *seed;           // dL/d(depth at gauge g after this step), n_gauges values (device)
    T *scratch;                   // scheme options only: 11 planes of pitch x (ny + 1) elements (face
                                  // contributions of both axes and the clip mask); null otherwise
    float2 *in_log;               // FP32, Eq. 3 as printed: per inflow slot, the adjoint of the cell's unclipped
                                  // depth and lambda_q of the face at this step, for pass 3
                                  // (launch_adjoint_inflow); null without inflow sections
    double *gn_in;                // FP64 and scheme options: the sections' dL/dn terms by slot (launch_gn_inflow_add)
};
template <typename T>
cudaError_t launch_adjoint_step(const AdjArgs<T> &a, cudaStream_t st);
// Pass 3 of the FP32 sweep (Eq. 3 as printed): the inflow sections' dL/dn terms of n_entries logged steps,
// entry e the global step first_step - e, summed per section cell into gn_in (added to gn after the sweep,
// launch_gn_inflow_add).
struct AdjInflowArgs {
    Geom geo;
    const InflowSec *secs;
    const int64_t *cells;
    const float *z, *n;
    int n_sec, n_slots, E;
    int64_t e0, first_step;       // epoch of the logs' first slice, step of entry 0
    int n_entries;
    const float *inflow_q;        // per epoch: E x n_slots
    const double *inflow_Q, *inflow_W, *dt;   // per epoch: nQ = E x n_sec values, one dt
    size_t nQ;
    const float2 *log;            // n_entries x n_slots
    double *terms;                // n_entries x n_slots (scratch)
    double *gn_in;                // n_slots
};
cudaError_t launch_adjoint_inflow(const AdjInflowArgs &A, cudaStream_t st);
// 2D tensor map (a CUtensorMap, 64-byte aligned storage at map) of a pitched FP32
// field of width x height elements and a row pitch of `pitch` elements, for boxes
// of box_w x box_h elements; elements outside the field read as zeros.
cudaError_t encode_map_f32(void *map, const float *base, int width, int height, int pitch, int box_w, int box_h);
// dst (pitched, precision T) = gn (pitched doubles).
template <typename T>
cudaError_t launch_gn_out(const Geom &g, const double *gn, T *dst, cudaStream_t st);
// The sections' terms gn_in (by slot) into gn, section by section.
cudaError_t launch_gn_inflow_add(double *gn, const double *gn_in, const InflowSec *secs, const int64_t *sec_cells, int n_sec,
                                 cudaStream_t st);

// Pitch padding (columns [cols, pitch) of rows x pitch elements of esz bytes):
// fill with the poison pattern, or count the elements whose bits differ from it.
cudaError_t launch_padding(void *a, size_t esz, int rows, int cols, int pitch, bool fill,
                           unsigned long long *count, cudaStream_t st);

// One thread waits budget_ns of device time on an mbarrier nothing arrives at;
// *gave_up (device) = 1 when the bounded wait gave up (the expected outcome).
cudaError_t launch_wait_probe(uint64_t budget_ns, int *gave_up, cudaStream_t st);

// The same from rows of depths (StepArgs::gauge_rows) of n_steps steps into out[n_steps][G].
cudaError_t launch_gauge_rows(const Geom &g, const float *rows, int n_rows, const int *row, const int64_t *cells, int G,
                              int n_steps, double *out, cudaStream_t st);
// Gather h at gauge cells into out[0..G).
template <typename T>
cudaError_t launch_gauges(const Geom &g, const T *h, const int64_t *cells, int G, double *out,
                          cudaStream_t st);

}  // namespace flood
