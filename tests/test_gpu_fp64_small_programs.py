"""FP64 products of few rows, few columns or short k in batches that fill the GPU
with a warp each: sizes on both sides of what a small program holds at once
(256 real, 128 complex outputs), of four times that, and of the k up to which it
takes them; smaller batches on both sides of where the shortest go to it; fixed and grouped calls with padded leading dimensions, alpha and
beta, and Hermitian updates. What a call leaves alone (padding, the upper
triangle) holds NaN.

Tolerance: sums of k products in FP64 in either order, alpha and beta: a
component differs by at most 2 (k + 4) u of |alpha| |a| |b| + |beta| |c| per real
product, four of them in a complex one (u = 2^-53).
"""
import numpy as np
import pytest

import paper_2203_09353_gb300 as bg

from gpu_util import dev, host

pytestmark = pytest.mark.gpu

U = 2.0 ** -53
COUNT = 2500  # (eight to a CTA, two CTAs per SM)

REAL = [(1, 256, 17), (1, 257, 16), (1, 300, 17), (300, 1, 16), (2, 200, 16), (1, 1024, 3),
        (1, 1025, 3), (3, 150, 8), (150, 3, 9), (5, 100, 8), (8, 64, 4), (8, 64, 5), (20, 20, 4),
        (32, 32, 4), (32, 32, 5), (33, 31, 4), (16, 64, 1), (29, 35, 2)]
COMPLEX = [(1, 128, 33), (1, 129, 32), (1, 300, 33), (300, 1, 32), (2, 200, 32), (1, 512, 3),
           (1, 513, 3), (3, 80, 8), (80, 3, 9), (16, 16, 8), (16, 16, 9), (32, 16, 8), (22, 23, 5)]


def values(rng, shape, dtype):
    x = rng.uniform(-1, 1, shape)
    return x + 1j * rng.uniform(-1, 1, shape) if dtype == "c128" else x


# (six to an SM of 152 up to k = 4, four of one or two rows or columns up to k = 8)
FEW = [("r64", (1, 300, 8), 607), ("r64", (1, 300, 8), 608), ("r64", (300, 1, 9), 1000),
       ("r64", (2, 150, 8), 700), ("r64", (8, 64, 4), 911), ("r64", (8, 64, 4), 912),
       ("r64", (32, 32, 2), 1000), ("c128", (1, 300, 8), 610), ("c128", (16, 16, 4), 912)]


@pytest.mark.parametrize("grouped", [False, True])
@pytest.mark.parametrize("dtype,size,count", [("r64", s, COUNT) for s in REAL] +
                         [("c128", s, COUNT) for s in COMPLEX] + FEW)
def test_product(gpu, dtype, size, count, grouped):
    (m, n, k), rng = size, np.random.default_rng(sum(size))
    lda, ldb, ldc = m + 1, k + 2, m + 3
    A, B = values(rng, (count, k, lda), dtype), values(rng, (count, n, ldb), dtype)
    C0 = values(rng, (count, n, ldc), dtype)
    C0[:, :, m:] = np.nan
    C = dev(C0)
    alpha, beta = (0.5 - 0.75j, 0.25 + 1j) if dtype == "c128" else (-0.75, 0.5)
    if grouped:
        rows = [(m, n, k, lda, ldb, ldc, i * lda * k, i * ldb * n, i * ldc * n)
                for i in range(count)]
        plan = bg.batched_gemm_plan(dtype, np.array(rows), None)
        bg.batched_gemm_grouped(plan, dev(A), dev(B), C, alpha, beta)
    else:
        bg.batched_gemm_fixed(dtype, m, n, k, alpha, dev(A), lda, lda * k, dev(B), ldb, ldb * n,
                              beta, C, ldc, ldc * n, count)
    got = host(C)
    a, b = A[:, :, :m].transpose(0, 2, 1), B[:, :, :k].transpose(0, 2, 1)
    c = C0[:, :, :m].transpose(0, 2, 1)
    bound = abs(alpha) * (np.abs(a) @ np.abs(b)) + abs(beta) * np.abs(c)
    err = np.abs(got[:, :, :m].transpose(0, 2, 1) - (alpha * (a @ b) + beta * c))
    assert np.all(err <= 8 * (k + 4) * U * bound)
    assert np.isnan(got[:, :, m:].real).all()


@pytest.mark.parametrize("dtype,n,k", [("r64", 17, 4), ("r64", 32, 4), ("r64", 31, 3),
                                       ("c128", 12, 8), ("c128", 16, 8), ("c128", 22, 7)])
def test_hermitian_update(gpu, dtype, n, k):
    rng = np.random.default_rng(n * k)
    A = values(rng, (COUNT, k, n), dtype)
    C = dev(np.full((COUNT, n, n), np.nan, dtype=A.dtype))
    rows = [(n, n, k, n, k, n, i * n * k, i * n * k, i * n * n) for i in range(COUNT)]
    plan = bg.batched_gemm_plan(dtype, np.array(rows), None, bg.BG_PLAN_HERK)
    bg.batched_gemm_grouped(plan, dev(A), None, C, 1.0, 0.0)
    got = host(C).transpose(0, 2, 1)
    a = A.transpose(0, 2, 1)
    ref, bound = a @ a.conj().transpose(0, 2, 1), np.abs(a) @ np.abs(a).transpose(0, 2, 1)
    low = np.tril(np.ones((n, n), dtype=bool))
    assert np.all((np.abs(got - ref) <= 8 * (k + 4) * U * bound)[:, low])
    assert np.isnan(got[:, ~low].real).all()
    assert np.all(got[:, np.arange(n), np.arange(n)].imag == 0)
