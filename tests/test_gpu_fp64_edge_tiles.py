"""Real FP64 products whose even split is the full 64 x 64 tile and whose last
tile is a row or a column short of it (127 = 64 + 63, 191 = 64 + 64 + 63, ...),
in batches on both sides of where the full tile is taken: fixed and grouped
calls, Hermitian updates and a chain step. C holds NaN before the call, which
an output left unwritten keeps.

Tolerance: both sides sum k products in FP64 in some order, so a component
differs by at most 2 k u sum |a||b| (u = 2^-53); 4 (k + 4) u sum |a||b| leaves
room for the rounding of alpha.
"""
import numpy as np
import pytest

import paper_2203_09353_gb300 as bg

from gpu_util import dev, host

pytestmark = pytest.mark.gpu

U = 2.0 ** -53


def close(got, a, b):
    return np.all(np.abs(got - a @ b) <= 4 * (a.shape[1] + 4) * U * (np.abs(a) @ np.abs(b)))


@pytest.mark.parametrize("m,n,batches", [
    (127, 127, (30, 31, 100)), (64, 127, (60, 61)), (127, 128, (31,)), (191, 128, (20, 21)),
    (255, 255, (7, 8)), (511, 511, (6, 7)), (1023, 1023, (1, 2))])
def test_fixed(gpu, m, n, batches):
    k, rng = n, np.random.default_rng(m + n)
    for batch in batches:
        A, B = rng.uniform(-1, 1, (batch, k, m)), rng.uniform(-1, 1, (batch, n, k))
        C = dev(np.full((batch, n, m), np.nan))
        bg.batched_gemm_fixed("r64", m, n, k, 1.0, dev(A), m, m * k, dev(B), k, k * n, 0.0, C, m,
                              m * n, batch)
        got = host(C)
        for i in {0, batch // 2, batch - 1}:
            assert close(got[i].T, A[i].T, B[i].T), (batch, i)
        assert not np.isnan(got).any(), batch


@pytest.mark.parametrize("n,count", [(127, 78), (191, 35), (255, 20), (511, 5), (1023, 2)])
@pytest.mark.parametrize("herk", [False, True])
def test_grouped(gpu, n, count, herk):
    k, ld, rng = 70, n + 1, np.random.default_rng(n)
    rows = [(n, n, k, ld, k, ld, i * ld * k, i * k * n, i * ld * n) for i in range(count)]
    A, B = rng.uniform(-1, 1, (count, k, ld)), rng.uniform(-1, 1, (count, n, k))
    C = dev(np.full((count, n, ld), np.nan))
    plan = bg.batched_gemm_plan("r64", np.array(rows), None, bg.BG_PLAN_HERK if herk else 0)
    bg.batched_gemm_grouped(plan, dev(A), None if herk else dev(B), C, 1.0, 0.0)
    got = host(C)
    keep = np.tril(np.ones((n, n), dtype=bool)) if herk else np.ones((n, n), dtype=bool)
    for i in range(count):
        a = A[i].T[:n]
        g = got[i].T
        assert close(np.where(keep, g[:n], a @ a.T if herk else 0.0), a, a.T if herk else B[i].T), i
        assert np.isnan(g[n:]).all() and np.isnan(g[:n][~keep]).all()


@pytest.mark.parametrize("n,walkers", [(127, 78), (255, 20)])
def test_chain_step(gpu, n, walkers):
    rng = np.random.default_rng(n)
    pool, states = rng.uniform(-1, 1, (3, n, n)), rng.uniform(-1, 1, (walkers, n, n))
    idx = rng.integers(0, 3, (1, walkers)).astype(np.int32)
    plan = bg.chain_plan("r64", [n] * walkers, np.arange(walkers) * n * n, [n] * 3,
                         np.arange(3) * n * n, None)
    pong = dev(np.full((walkers, n, n), np.nan))
    bg.chain_step(plan, dev(pool), dev(idx), dev(states), pong, 1)
    got = host(pong)
    for w in range(walkers):
        assert close(got[w].T, pool[idx[0, w]].T, states[w].T), w
