"""flood_coarsen's row vectors: every vector width and alignment, the general kernel's
factors, and blocks whose float sums overflow, against NumPy.  FP32 block means are
correctly rounded up to the last place (1.2e-7), FP64 sums differ by their order (1e-15).
"""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def F():
    import paper_2204_10323_gb300 as F
    return F


def block_mean(z, f):
    my, mx = -(-z.shape[0] // f), -(-z.shape[1] // f)
    return np.array([[z[j * f:(j + 1) * f, i * f:(i + 1) * f].astype(np.float64).mean() for i in range(mx)] for j in range(my)])


@pytest.mark.parametrize("dtype,rtol", [(np.float32, 1.2e-7), (np.float64, 1e-15)])
@pytest.mark.parametrize("nx,ny,f", [(64, 32, 4), (62, 9, 2), (64, 17, 8), (63, 20, 4), (48, 33, 3), (100, 41, 5),
                                     (64, 40, 16), (70, 40, 17), (33, 7, 1), (10, 6, 20)])
@pytest.mark.parametrize("skip", [0, 1])
def test_coarsen_vectors(nx, ny, f, dtype, rtol, skip):
    import torch
    Fm = F()
    z = np.random.default_rng(nx + f).normal(1.0, 30.0, (ny, nx)).astype(dtype) + dtype(40.0)
    buf = torch.zeros(z.size + skip, dtype=torch.float32 if dtype == np.float32 else torch.float64, device="cuda")
    t = buf[skip:].view(ny, nx)
    t.copy_(torch.from_numpy(z))
    np.testing.assert_allclose(Fm.coarsen(t, f).cpu().numpy(), block_mean(z, f).astype(dtype), rtol=rtol)


def test_coarsen_of_infinite_and_huge_cells():
    # the float pair overflows where the double sum does not; infinities and NaN stay in their blocks
    Fm = F()
    z = np.full((8, 12), 3e38, np.float32)
    z[0, 4], z[1, 9], z[5, 0], z[5, 1] = np.inf, np.nan, np.inf, -np.inf
    got = Fm.coarsen(z, 4)
    want = np.float32([[3e38, np.inf, np.nan], [np.nan, 3e38, 3e38]])
    np.testing.assert_allclose(got, want, rtol=1.2e-7)
