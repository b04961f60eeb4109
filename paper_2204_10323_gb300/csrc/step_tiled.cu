// step_tiled.cu -- the temporal-blocking kernels (step_tiled.cuh) for Eq. 3 as
// printed, the host-side split of a grid into (chunk, strip) work items, and
// the launchers, which send the scheme options to step_tiled_opts.cu.
#include "step_tiled.cuh"

namespace flood {

int sm_count()
{
    static const int n = [] {
        int dev = 0, v = 0;
        if (cudaGetDevice(&dev) == cudaSuccess && cudaDeviceGetAttribute(&v, cudaDevAttrMultiProcessorCount, dev) == cudaSuccess && v > 0)
            return v;
        (void)cudaGetLastError();
        return 152;
    }();
    return n;
}

int tiled_resident(int mode) { return sm_count() * tiled_warps(mode); }

// Rows per item.  An item of r rows takes r + 2K ticks; a tick of a warp alone on its quarter of an SM
// takes about 1650 cycles, beside others about 1150 + 490 per warp (K = 4, measured with the clock
// register at 1024^2 .. 4096^2), and 1000 more in an edge strip, whose items are therefore shorter.  The
// rows minimise the waves of items, the last one with the warps it has: few rows fill the GPU evenly but
// repeat 2K rows each.  us per step with rows chosen so / fixed at 96: 11.0 / 36.8 (1024^2), 15.9 / 37.3
// (2048^2), 39 / 50 (4096^2), 131 / 131 (8192^2), 465 / 477 (16384^2); with the higher beds kept and
// dependent launches since then 8.2, 13.4, 39, 120 and 463.
void tiled_rows(int nx, int ny, int K, int mode, int *rows, int *rows_edge)
{
    const int out = out_cols(K, mode);
    tiled_rows_for((nx + out - 1) / out, ny, 2 * K, tiled_warps(mode), 1150.0, 490.0, 1000.0, rows, rows_edge);
}

// The rule for items of r + `repeat` ticks, `warps` of them per SM, a tick taking base + slope * (warps on a
// quarter of an SM), and `edge` more in an edge strip.
void tiled_rows_for(int n_strips, int ny, int repeat, int warps, double base, double slope, double edge_more, int *rows,
                    int *rows_edge)
{
    static constexpr int kTry[] = {2,  3,  4,  6,  8,  10, 12, 14, 16,  18,  20,  22,  24,  28,  32, 36,
                                   40, 44, 48, 56, 64, 80, 96, 112, 128, 144, 160, 192, 256};
    const int sms = sm_count(), resident = sms * warps, n_edge = n_strips < 2 ? n_strips : 2;
    const auto tick = [&](double w) { return base + slope * (w > 1.0 ? w : 1.0); };
    const auto even = [&](int r) { return (ny + (ny + r - 1) / r - 1) / ((ny + r - 1) / r); };   // equal chunks of at most r
    double best = -1.0;
    for (int t : kTry) {
        if (t < repeat / 2 && t < ny) continue;        // rows that an item mostly repeats
        const int r = even(t), re = even((5 * t + 7) / 8);
        const long long n = (long long)n_edge * ((ny + re - 1) / re) + (long long)(n_strips - n_edge) * ((ny + r - 1) / r);
        const long long full = n / resident, rest = n % resident;
        double cost = (r + repeat) * (full * tick(warps / 4.0) + (rest ? tick(rest / (4.0 * sms)) : 0.0));
        const double edge = (re + repeat) * (tick(full ? warps / 4.0 : rest / (4.0 * sms)) + edge_more);
        if (edge > cost) cost = edge;
        if (best < 0.0 || cost < best) {
            best = cost;
            *rows = r;
            *rows_edge = re;
        }
        if (t >= ny) break;
    }
}

// Row chunks for the items of a grid of n_strips strips and ny rows on `resident` pipelines that walk
// them in turn (a caller's cap on the pipelines): the chunk count minimises the ticks of the busiest
// pipeline, (items per pipeline) x (chunk rows + 3K - 1).  (An item runs 2K ticks more than it has rows by now; callers of
// flood_debug_tiled_split rely on the values of this form, and the choice between them is a matter of a per cent.)
static void tiled_split(int n_strips, int ny, int resident, int K, int *chunk_rows, int *blocks)
{
    static thread_local int memo[4] = {-1, -1, -1, -1}, memo_rows = 0;   // per thread: no race between handles
    if (memo[0] == n_strips && memo[1] == ny && memo[2] == resident && memo[3] == K) {
        const long long items = (long long)n_strips * ((ny + memo_rows - 1) / memo_rows);
        *chunk_rows = memo_rows;
        *blocks = (int)(items < resident ? items : resident);
        return;
    }
    long long best = -1;
    int best_rows = ny;
    const int max_chunks = (ny + 15) / 16;            // chunks of at least 16 rows
    for (int c = 1; c <= max_chunks; c++) {
        const int rows = (ny + c - 1) / c;
        const int chunks = (ny + rows - 1) / rows;
        const long long items = (long long)n_strips * chunks;
        const long long waves = (items + resident - 1) / resident;
        const long long ticks = waves * (rows + 3 * K - 1);
        if (best < 0 || ticks < best) {
            best = ticks;
            best_rows = rows;
        }
    }
    memo[0] = n_strips;
    memo[1] = ny;
    memo[2] = resident;
    memo[3] = K;
    memo_rows = best_rows;
    const long long items = (long long)n_strips * ((ny + best_rows - 1) / best_rows);
    *chunk_rows = best_rows;
    *blocks = (int)(items < resident ? items : resident);
}

// The same with about eight items per pipeline of at least 24 K rows, so that the launch ends
// evenly; a grid that would get fewer than four such items per pipeline keeps the split above.
void tiled_split_dynamic(int n_strips, int ny, int resident, int K, int *chunk_rows, int *blocks)
{
    const long long target = 8LL * resident;
    const long long chunks = (target + n_strips - 1) / n_strips;
    int rows = (int)((ny + chunks - 1) / chunks);
    const int min_rows = 24 * K;
    if (rows < min_rows) {
        rows = min_rows;
        if ((long long)n_strips * ((ny + rows - 1) / rows) < 4LL * resident) {
            tiled_split(n_strips, ny, resident, K, chunk_rows, blocks);
            return;
        }
    }
    const long long items = (long long)n_strips * ((ny + rows - 1) / rows);
    *chunk_rows = rows;
    *blocks = (int)(items < resident ? items : resident);
}

int tiled_items(const Geom &g, int rows, int rows_edge, int k_steps)
{
    const int mode = (g.theta != 1.0 ? 1 : 0) | (g.friction != 0 ? 2 : 0);
    return tiled_item_count(g.nx, g.ny, out_cols(k_steps, mode), rows, rows_edge);
}

// Scheme mode of a grid: bit 0 theta weighting, bit 1 vector-norm friction.
static int tiled_mode(const Geom &g) { return (g.theta != 1.0 ? 1 : 0) | (g.friction != 0 ? 2 : 0); }

// step_tiled_opts.cu: the same launchers for modes 1..3.
cudaError_t launch_step_tiled_opts(const StepArgs<float> &a, int mode, cudaStream_t st);
cudaError_t launch_step_tiled_ensemble_opts(const GridTable &t, int k_steps, int s0, int want_hmax, int mode, cudaStream_t st);

cudaError_t launch_step_tiled_ensemble(const GridTable &t, int k_steps, int s0, int want_hmax, int mode, cudaStream_t st)
{
    if (mode != 0) return launch_step_tiled_ensemble_opts(t, k_steps, s0, want_hmax, mode, st);
    return launch_tiled_ensemble_mode<0>(t, k_steps, s0, want_hmax, st);
}

cudaError_t launch_step_tiled(const StepArgs<float> &a, cudaStream_t st)
{
    const int mode = tiled_mode(a.geo);
    if (mode != 0) return launch_step_tiled_opts(a, mode, st);
    return launch_tiled_mode<0>(a, st);
}

}  // namespace flood

#include "flood.h"

extern "C" flood_status flood_debug_tiled_split(int32_t nx, int32_t ny, int32_t k_steps, int32_t mode,
                                                int32_t resident, int32_t *chunk_rows, int32_t *blocks,
                                                int32_t *n_items)
{
    using namespace flood;
    if (nx < 1 || ny < 1 || !(k_steps >= 1 && (k_steps <= 4 || k_steps == 8)) || mode < 0 || mode > 3 ||
        resident < 1 || !chunk_rows || !blocks || !n_items)
        return FLOOD_ERR_ARG;
    const int out = out_cols(k_steps, mode);
    const int n_strips = (nx + out - 1) / out;
    int rows = 0, b = 0;
    tiled_split_dynamic(n_strips, ny, resident, k_steps, &rows, &b);
    const long long items = (long long)n_strips * ((ny + rows - 1) / rows);
    if (items > 0x7fffffffLL) return FLOOD_ERR_ARG;
    *chunk_rows = rows;
    *blocks = b;
    *n_items = (int32_t)items;
    return FLOOD_OK;
}
