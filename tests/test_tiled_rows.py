"""Rows per work item that the temporal-blocking kernel takes by itself, computed by the library's host code (no GPU):
the items cover every cell once, and an ensemble's rows are those that its cost rule gives for the warps that a GPU of
152 multiprocessors holds of the scheme's kernel (8 a multiprocessor with the theta weighting, else 12).
"""
import math

import pytest

EDGE = lambda r: (5 * r + 7) // 8


def F():
    import paper_2204_10323_gb300 as F
    return F


def width(K, mode):
    return 116 if K == 4 and mode & 1 else 120


@pytest.mark.parametrize("K,mode", [(4, 0), (4, 1), (4, 2), (4, 3), (3, 1), (2, 0), (1, 2)])
def test_items_cover_the_grid(K, mode):
    shapes = [(1, 1), (7, 5), (120, 3), (121, 300), (300, 40), (1024, 1024), (1500, 701), (2048, 2048), (4096, 4096),
              (16384, 16384), (3, 600000), (100000, 2)]
    for (nx, ny), (rows, edge, items) in zip(shapes, F().flood_debug_tiled_rows(shapes, K, mode)):
        assert 1 <= rows <= ny and 1 <= edge <= ny
        strips = math.ceil(nx / width(K, mode))
        n_edge = min(strips, 2)
        assert items == n_edge * math.ceil(ny / edge) + (strips - n_edge) * math.ceil(ny / rows)
        # as the kernel numbers them: edge strips first
        if items > 5000:
            continue
        seen = {}
        edge_items = n_edge * math.ceil(ny / edge)
        for i in range(items):
            if i < edge_items:
                s, r, y0 = (strips - 1 if i % n_edge else 0), edge, i // n_edge * edge
            else:
                k = i - edge_items
                s, r, y0 = 1 + k % (strips - n_edge), rows, k // (strips - n_edge) * rows
            seen.setdefault(s, []).append((y0, min(y0 + r, ny)))
        assert sorted(seen) == list(range(strips))
        for chunks in seen.values():
            chunks.sort()
            assert chunks[0][0] == 0 and chunks[-1][1] == ny
            assert all(a[1] == b[0] for a, b in zip(chunks, chunks[1:]))


def ensemble_rows(shapes, K, mode, most):
    def rows_of(b, nx, ny):
        return min(max(int(b * math.sqrt(nx * ny / 2.0 ** 20) + 0.5), 8), ny)

    def cost(b):
        ticks = longest = 0.0
        for nx, ny in shapes:
            r = rows_of(b, nx, ny)
            strips = math.ceil(nx / width(K, mode))
            e = min(strips, 2)
            ticks += (e * math.ceil(ny / EDGE(r)) + (strips - e) * math.ceil(ny / r)) * (r + 2 * K)
            longest = max(longest, r + 2.0 * K)
        return max(ticks / (152 * (8 if mode & 1 else 12)), longest) + 0.1 * longest
    tries = [b for b in (8, 12, 16, 20, 24, 32, 40, 48, 64, 80, 96, 128, 160, 192, 256, 320, 384, 512, most) if b <= most]
    best = min(tries, key=cost)
    return [rows_of(best, *s) for s in shapes]


@pytest.mark.parametrize("mode", [0, 1, 2, 3])
@pytest.mark.parametrize("members", [1, 3, 5, 12, 20, 40])
def test_ensembles_count_the_warps_of_their_scheme(members, mode):
    sizes = [(256, 256), (512, 512), (1024, 1024), (1536, 1024), (2048, 2048), (333, 777)]
    shapes = [sizes[k % 6] for k in range(members)]
    for most in (7, 64, 512):
        got = F().flood_debug_tiled_rows(shapes, 4, mode, most)
        assert [g[0] for g in got] == ensemble_rows(shapes, 4, mode, most)
        assert [g[1] for g in got] == [EDGE(g[0]) for g in got]


def test_theta_scenarios_take_longer_items_than_as_printed():
    shapes = [(256, 256), (512, 512), (1024, 1024)]
    plain, theta = (F().flood_debug_tiled_rows(shapes, 4, mode, 512) for mode in (0, 1))
    assert theta[2][0] > plain[2][0]


@pytest.mark.parametrize("args", [([], 4, 0, 0), ([(0, 5)], 4, 0, 0), ([(5, 5)], 5, 0, 0), ([(5, 5)], 4, 4, 0), ([(5, 5)], 4, 0, -1),
                                  ([(1 << 24, 1 << 24)], 4, 0, 0)])
def test_bad_arguments(args):
    Fm = F()
    with pytest.raises(Fm.FloodError):
        Fm.flood_debug_tiled_rows(*args)
