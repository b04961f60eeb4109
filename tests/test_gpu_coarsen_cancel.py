"""Single-precision block means, also where a block's cells cancel: opposite huge cells, sums next to zero, blocks of
one sign, tiny and subnormal cells, against exact rational means.  Tolerance: the rounding of the result (half a unit in
the last place), 2^-7 of a unit for a sum as a float pair, and for a sum in double the rounding of its additions, 2^-53
of the magnitudes' sum each."""
from fractions import Fraction

import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def exact_mean(block):
    return Fraction(sum(map(Fraction, block.ravel().tolist()), Fraction(0)) / block.size)


def cancelling(rng, ny, nx, f):
    z = rng.uniform(0.2, 0.4, (ny, nx))
    for j in range(0, ny, f):
        for i in range(0, nx, f):
            b = z[j:j + f, i:i + f]
            at = rng.permutation(b.size)[:2]
            if b.size > 1:
                b.flat[at[0]], b.flat[at[1]] = 1e8, -1e8
    return z


def balanced(rng, ny, nx, f):
    z = rng.standard_normal((ny, nx)).astype(np.float32)
    z[:, 1::2] = -z[:, 0:nx - nx % 2:2] * np.float32(1 + 2.0 ** -20)
    return z


@pytest.mark.parametrize("f", [2, 3, 4, 5, 8, 12, 16])
@pytest.mark.parametrize("kind", ["cancelling", "balanced", "one_sign", "tiny", "subnormal", "zero"])
def test_block_means_are_exact(kind, f):
    import torch
    import paper_2204_10323_gb300 as Fm
    rng = np.random.default_rng(f)
    ny, nx = 3 * f + 1, 4 * f
    z = {"cancelling": lambda: cancelling(rng, ny, nx, f), "balanced": lambda: balanced(rng, ny, nx, f),
         "one_sign": lambda: rng.uniform(0.0, 40.0, (ny, nx)), "tiny": lambda: rng.standard_normal((ny, nx)) * 1e-33,
         "subnormal": lambda: rng.standard_normal((ny, nx)) * 1e-41, "zero": lambda: np.zeros((ny, nx))}[kind]()
    z = z.astype(np.float32)
    got = Fm.coarsen(torch.from_numpy(z).cuda(), f).cpu().numpy()
    for J in range(got.shape[0]):
        for I in range(got.shape[1]):
            want = exact_mean(z[J * f:(J + 1) * f, I * f:(I + 1) * f])
            unit = Fraction(float(np.spacing(np.float32(abs(float(want))))))
            size = sum((abs(Fraction(v)) for v in z[J * f:(J + 1) * f, I * f:(I + 1) * f].ravel().tolist()), Fraction(0))
            assert abs(Fraction(float(got[J, I])) - want) <= unit * Fraction(65, 128) + size / 2 ** 53, (J, I, float(want), got[J, I])
