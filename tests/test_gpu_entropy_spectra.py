"""Eigenvalues and entropies of states with prescribed Schmidt spectra, at the
edges of the reduction and the bisection: orders from 2 to 1024 (one CTA and
several to a walker, all columns in shared memory and only the last ones), 3 to
129 walkers (each number of lanes to an eigenvalue), spectra that are flat,
clustered, low-rank, geometric, and states of extreme scale.

Tolerance: a backward-stable reduction and bisection move an eigenvalue by at
most 4 K u ||G|| (u = 2^-53; the largest eigenvalue bounds ||G||), and the Gram
matrix's K-term sums and the test's own construction of the state by as much
again. Each -p ln p then moves by that times 1 + |ln| of it, K of them.
"""
import numpy as np
import pytest

import paper_2203_09353_gb300 as bg

pytestmark = pytest.mark.gpu

U = 2.0 ** -53


def haar(rng, n):
    z = rng.standard_normal((n, n)) + 1j * rng.standard_normal((n, n))
    q, r = np.linalg.qr(z)
    return q * (np.diag(r) / np.abs(np.diag(r)))


def spectra(rng, K):
    k = np.arange(K)
    return [rng.random(K) + 0.01, np.ones(K), 0.5 ** np.minimum(k, 200.0),
            np.where(k < 3, 1.0 + k, 0.0), np.where(k < 1, 1.0, 0.0),
            1.0 + 1e-13 * rng.random(K), np.repeat(rng.random(K // 2 + 1), 2)[:K]]


@pytest.mark.parametrize("slices", [0, 9])
@pytest.mark.parametrize("split,spins,walkers", [
    (1, 2, 3), (2, 5, 200), (4, 8, 129), (6, 12, 3), (6, 13, 16), (6, 12, 40), (6, 12, 80),
    (6, 12, 129), (7, 14, 7), (8, 16, 9), (9, 18, 4), (10, 20, 2)])
def test_spectra(gpu, slices, split, spins, walkers):
    import torch
    rng = np.random.default_rng(100 * spins + split)
    K, M = 1 << split, 1 << (spins - split)
    Um, V = haar(rng, M)[:, :K], haar(rng, K)
    all_p = [p / p.sum() for p in spectra(rng, K)]
    states = [((Um * np.sqrt(p)) @ V.conj().T).reshape(-1) for p in all_p]
    scale = [1.0, 1e-140, 1e120]
    psi = np.stack([states[w % len(states)] * scale[w % 3] for w in range(walkers)])
    plan = bg.entropy_plan(walkers, spins, split,
                           prec=bg.precision("split", slices) if slices else None)
    ent = torch.zeros(walkers, dtype=torch.float64, device="cuda")
    eig = torch.zeros(walkers, K, dtype=torch.float64, device="cuda")
    bg.batched_entropy(plan, torch.from_numpy(psi).cuda(), ent, eig)
    bg.check_device_errors()
    ent, eig = ent.cpu().numpy(), eig.cpu().numpy()
    for w in range(walkers):
        p = np.sort(all_p[w % len(states)])
        tol = 8 * K * U * p[-1]
        got = eig[w] / scale[w % 3] ** 2
        assert np.all(np.diff(eig[w]) >= 0)
        assert np.max(np.abs(got - p)) <= tol, w
        want = -np.sum(p[p > 0] * np.log(p[p > 0]))
        assert abs(ent[w] - want) <= K * tol * (1 - np.log(tol)), w
    plan.close()


def test_zero_and_not_finite(gpu):
    """A zero state has entropy 0; a NaN or infinite amplitude gives NaN, for its walker alone."""
    import torch
    rng = np.random.default_rng(1)
    psi = rng.standard_normal((4, 512)) + 1j * rng.standard_normal((4, 512))
    psi[0] = 0.0
    psi[1, 7] = np.nan
    psi[2, 300] = np.inf
    ent = torch.zeros(4, dtype=torch.float64, device="cuda")
    eig = torch.zeros(4, 16, dtype=torch.float64, device="cuda")
    plan = bg.entropy_plan(4, 9, 4)
    bg.batched_entropy(plan, torch.from_numpy(psi).cuda(), ent, eig)
    ent, eig = ent.cpu().numpy(), eig.cpu().numpy()
    assert ent[0] == 0.0 and not eig[0].any()
    assert np.isnan(ent[1]) and np.isnan(ent[2])
    p = np.linalg.svd(psi[3].reshape(-1, 16), compute_uv=False) ** 2
    p /= p.sum()
    t = 8 * 16 * U
    assert abs(ent[3] + np.sum(p * np.log(p))) <= 16 * t * (1 - np.log(t))
    plan.close()
