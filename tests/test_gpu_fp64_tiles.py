"""The FP64 tiles at the edges of their dispatch: one output to a full tile and
one past it, batches that spread an instance over many CTAs and batches that
do not, in fixed and grouped calls, Hermitian updates included.

Tolerance: both sides sum k products in FP64, in ascending order; the kernel
contracts each into an FMA, the oracle rounds twice, so a component differs
by at most 2 k u sum |a||b| (u = 2^-53), plus the few roundings of alpha and
beta: 4 (k + 4) u (|alpha| sum |a||b| + |beta||c|), four times that for the
complex products' two terms each.
"""
import numpy as np
import pytest

import paper_2203_09353_gb300 as bg

from gpu_util import dev, host

pytestmark = pytest.mark.gpu

U = 2.0 ** -53


def draw(rng, shape, dtype):
    x = rng.uniform(-1, 1, shape)
    return x + 1j * rng.uniform(-1, 1, shape) if dtype == "c128" else x


def bound(a, b, c, alpha, beta, k, dtype):
    s = np.abs(a) @ np.abs(b)
    return (16 if dtype == "c128" else 4) * (k + 4) * U * (abs(alpha) * s + abs(beta) * np.abs(c))


@pytest.mark.parametrize("dtype", ["r64", "c128"])
@pytest.mark.parametrize("m,n,k,batch", [
    (1, 1, 3, 1), (31, 33, 17, 2), (32, 32, 16, 5), (32, 33, 31, 400), (64, 64, 64, 3),
    (64, 64, 15, 200), (64, 63, 16, 1), (65, 64, 33, 2), (16, 16, 16, 5000), (11, 23, 5, 2500),
    (1, 200, 9, 7), (129, 2, 70, 4)])
def test_fixed(gpu, dtype, m, n, k, batch):
    rng = np.random.default_rng(m * 7919 + n * 31 + k)
    A, B, C = (draw(rng, s, dtype) for s in ((batch, k, m), (batch, n, k), (batch, n, m)))
    alpha, beta = (0.5 - 1j, 0.75j) if dtype == "c128" else (-1.5, 0.25)
    Cd = dev(C)
    bg.batched_gemm_fixed(dtype, m, n, k, alpha, dev(A), m, m * k, dev(B), k, k * n, beta, Cd, m,
                          m * n, batch)
    got = host(Cd)
    for i in (range(batch) if batch < 50 else rng.integers(0, batch, 50)):
        a, b, c = A[i].T, B[i].T, C[i].T
        ref = alpha * (a @ b) + beta * c
        assert np.all(np.abs(got[i].T - ref) <= bound(a, b, c, alpha, beta, k, dtype)), i


@pytest.mark.parametrize("dtype", ["r64", "c128"])
@pytest.mark.parametrize("edge,count", [(20, 7), (40, 300), (150, 25)])
@pytest.mark.parametrize("herk", [False, True])
def test_grouped(gpu, dtype, edge, count, herk):
    rng = np.random.default_rng(edge + count)
    rows, off = [], [0, 0, 0]
    for _ in range(count):
        m, n, k = (int(x) for x in rng.integers(1, edge + 1, 3))
        if herk:
            m = n
        lda, ldb, ldc = m + int(rng.integers(0, 3)), k + 1, m + 2
        rows.append((m, n, k, lda, ldb, ldc, *off))
        for q, size in enumerate((lda * k, ldb * n, ldc * n)):
            off[q] += size
    A, B, C = (draw(rng, x, dtype) for x in off)
    plan = bg.batched_gemm_plan(dtype, np.array(rows), None, bg.BG_PLAN_HERK if herk else 0)
    Cd = dev(C)
    bg.batched_gemm_grouped(plan, dev(A), None if herk else dev(B), Cd, 2.0, -0.5)
    got = host(Cd)
    want_eq = np.ones(C.size, dtype=bool)
    for m, n, k, lda, ldb, ldc, ao, bo, co in rows:
        a = A[ao:ao + lda * k].reshape(k, lda).T[:m]
        b = a.conj().T if herk else B[bo:bo + ldb * n].reshape(n, ldb).T[:k]
        c = C[co:co + ldc * n].reshape(n, ldc).T[:m]
        g = got[co:co + ldc * n].reshape(n, ldc).T[:m]
        mask = np.tril(np.ones((m, n), dtype=bool)) if herk else np.ones((m, n), dtype=bool)
        ref, lim = 2.0 * (a @ b) - 0.5 * c, bound(a, b, c, 2.0, 0.5, k, dtype)
        if herk:
            np.fill_diagonal(ref, ref.diagonal().real)
        assert np.all((np.abs(g - ref) <= lim)[mask])
        w = want_eq[co:co + ldc * n].reshape(n, ldc).T[:m]
        w[mask] = False
    assert np.array_equal(got[want_eq], C[want_eq])
