"""Entropies of small orders on both sides of one walker per SM, from where on
the reduction packs several walkers to an SM and a warp takes a walker's sums:
orders 2 to 32 (and 64, which does neither), random, product and zero states.

Tolerance on an eigenvalue: 4 K u ||G|| for the reduction and the bisection,
as much for the library's eigensolver, and 2 M u ||G|| for each side's M-term
sums in G (u = 2^-53, M = K). -p ln p then moves by that times 1 + |ln| of it.
"""
import numpy as np
import pytest
import torch

import paper_2203_09353_gb300 as bg

from gpu_util import host

pytestmark = pytest.mark.gpu

U = 2.0 ** -53


@pytest.mark.parametrize("split", [1, 2, 3, 4, 5, 6])
@pytest.mark.parametrize("extra", [0, 1, 600])
def test_many_walkers(gpu, split, extra):
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    W, K, spins = sms + extra, 1 << split, 2 * split
    rng = np.random.default_rng(100 * split + extra)
    x = rng.standard_normal((2, W, K, K))
    X = x[0] + 1j * x[1]
    X[5] = np.outer(X[5, 0], X[5, 1])
    X[-2] = 0.0
    plan = bg.entropy_plan(W, spins, split)
    ent = torch.zeros(W, dtype=torch.float64, device="cuda")
    eig = torch.zeros(W * K, dtype=torch.float64, device="cuda")
    bg.batched_entropy(plan, torch.from_numpy(X.reshape(W, -1)).cuda(), ent, eig)
    only = torch.zeros_like(ent)
    bg.batched_entropy(plan, torch.from_numpy(X.reshape(W, -1)).cuda(), only)
    bg.check_device_errors()
    got, ent = host(eig).reshape(W, K), host(ent)
    lam = np.linalg.eigvalsh(np.swapaxes(X, 1, 2) @ X.conj())
    lim = 12 * K * U * lam[:, -1]
    assert np.all(np.abs(got - lam) <= lim[:, None])
    assert np.all(np.diff(got, axis=1) >= 0) and np.array_equal(ent, host(only))
    total = lam.sum(axis=1)
    p = np.clip(lam, 0, None) / np.where(total > 0, total, 1.0)[:, None]
    want = -np.sum(p * np.log(np.where(p > 0, p, 1.0)), axis=1)
    dp = 24 * K * U
    assert np.all(np.abs(ent - want) <= K * dp * (1 + abs(np.log(dp))))
