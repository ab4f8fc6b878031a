"""The split mode's tile kernel at the edges of its tiles: every tile width that
an instance's columns are dealt into, K from one element to several blocks of 64
with partial last steps (one block, the first and last of several, those between
take their planes in another order), several row blocks, batches beyond one wave.

The inputs are whole numbers up to 7 in magnitude: every slice count represents
them and their sums of products (below 2^53) exactly, so C is exact.
"""
import numpy as np
import pytest

import paper_2203_09353_gb300 as bg
from paper_2203_09353_gb300 import synth

from gpu_util import host, run_grouped

pytestmark = pytest.mark.gpu

WIDTHS = (1, 15, 16, 17, 31, 33, 47, 48, 49, 63, 64, 65, 79, 81, 95, 97, 113, 127, 129, 145, 200)


def whole(rng, size, dtype):
    x = rng.integers(-7, 8, size).astype(np.float64)
    return x + 1j * rng.integers(-7, 8, size) if dtype == "c128" else x


@pytest.mark.parametrize("dtype", ["r64", "c128"])
@pytest.mark.parametrize("slices", [1, 3, 4, 5, 6, 8, 9, 10, 12])
@pytest.mark.parametrize("k", [1, 63, 64, 65, 130, 250])
def test_widths(gpu, dtype, slices, k):
    rng = np.random.default_rng(slices * 1000 + k)
    shapes = [(int(rng.choice((65, 128, 131))), n, k) for n in WIDTHS]
    shapes += [(70, 40, k)] * 320 if k == 65 else []
    rows, off = [], [0, 0, 0]
    for m, n, kk in shapes:
        rows.append((m, n, kk, m, kk + 1, m + 3, *off))
        off = [off[0] + m * kk, off[1] + (kk + 1) * n, off[2] + (m + 3) * n]
    table = np.array(rows, dtype=np.int64)
    A, B, C = (whole(rng, o, dtype) for o in off)
    batch = synth.Batch("widths", dtype, table, A, B, C.copy(), 1.0, 2.0)
    got, _ = run_grouped(batch, bg.precision("split", slices), bg.BG_PLAN_SPLIT_TILES)
    got = host(got)
    for m, n, kk, lda, ldb, ldc, ao, bo, co in rows:
        a = A[ao:ao + lda * kk].reshape(kk, lda).T
        b = B[bo:bo + ldb * n].reshape(n, ldb).T[:kk]
        c = C[co:co + ldc * n].reshape(n, ldc).T[:m]
        g = got[co:co + ldc * n].reshape(n, ldc).T
        assert np.array_equal(g[:m], a @ b + 2.0 * c), (m, n, kk)
        assert np.array_equal(g[m:], C[co:co + ldc * n].reshape(n, ldc).T[m:])
