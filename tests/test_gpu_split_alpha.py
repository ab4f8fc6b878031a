"""Split mode, alpha a power of two: taken as an exponent and a sign, without a
multiply. Scaling by a power of two is exact, so C must be the alpha = 1 result
times alpha bit for bit, here with beta = 0 (signed zeros included), and within
one rounding of beta C + alpha A B otherwise.
"""
import numpy as np
import pytest

import paper_2203_09353_gb300 as bg
from paper_2203_09353_gb300 import synth

from gpu_util import host, run_grouped

pytestmark = pytest.mark.gpu


def batch(dtype, alpha, beta, seed):
    rng = np.random.default_rng(seed)
    rows, off = [], [0, 0, 0]
    for m, n, k in ((5, 9, 3), (33, 20, 64), (100, 70, 130), (129, 49, 65)):
        rows.append((m, n, k, m, k, m, *off))
        off = [off[0] + m * k, off[1] + k * n, off[2] + m * n]
    A, B, C = (rng.standard_normal(o) + (1j * rng.standard_normal(o) if dtype == "c128" else 0)
               for o in off)
    A[:5] = 0.0  # a row of zero products
    return synth.Batch("alpha", dtype, np.array(rows, dtype=np.int64), A, B, C, alpha, beta)


@pytest.mark.parametrize("dtype", ["r64", "c128"])
@pytest.mark.parametrize("slices", [3, 6, 9])
@pytest.mark.parametrize("alpha", [-1.0, 2.0, -0.5, 2.0 ** -200, -(2.0 ** 300)])
def test_power_of_two(gpu, dtype, slices, alpha):
    prec = bg.precision("split", slices)
    one, _ = run_grouped(batch(dtype, 1.0, 0.0, 3), prec)
    got, _ = run_grouped(batch(dtype, alpha, 0.0, 3), prec)
    one, got = (host(x).view(np.float64) for x in (one, got))
    assert np.array_equal((alpha * one).view(np.int64), got.view(np.int64))
    b = batch(dtype, alpha, 0.75, 3)
    both, _ = run_grouped(b, prec)
    c = 0.75 * b.C.view(np.float64)
    want = c + alpha * one  # (the kernel rounds once more or less: an fma)
    err = np.abs(host(both).view(np.float64) - want)
    assert np.all(err <= 2.0 ** -52 * (np.abs(c) + np.abs(alpha * one)))
