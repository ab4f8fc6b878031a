"""Eigenvalues of Gram matrices of every precision, on states of low entropy:
1 to 12 slices and short digits, which leave G indefinite by their own truncation
error, beside 9 slices and FP64. The plan's own G, from a Hermitian update of
the same precision, is the reference: the reduction and the bisection are
judged apart from the error of G.

Tolerance: a backward-stable reduction and bisection move an eigenvalue by at
most 4 K u ||G|| (u = 2^-53), the library eigensolver by as much again.
"""
import numpy as np
import pytest
import torch

import paper_2203_09353_gb300 as bg

from gpu_util import host

pytestmark = pytest.mark.gpu

U = 2.0 ** -53
PRECISIONS = [None] + [bg.precision("split", s) for s in range(1, 13)] + [
    bg.precision("split", 9, 2), bg.precision("split", 6, 3), bg.precision("split", 2, 4)]


def unitary(rng, n):
    return np.linalg.qr(rng.standard_normal((n, n)) + 1j * rng.standard_normal((n, n)))[0]


def states_of(rng, spins, split):
    M, K = 1 << (spins - split), 1 << split
    k = np.arange(K)
    out = []
    for p in (k < 1, k < 3, 0.5 ** np.minimum(k, 200.0), 0.1 ** np.minimum(k, 200.0), k < K // 2):
        out.append(unitary(rng, M)[:, :K] * np.sqrt(p / p.sum()) @ unitary(rng, K).conj().T)
    for noise in (0.0, 1e-4):  # product states of single spins
        psi = np.ones(1)
        for _ in range(spins):
            spin = rng.standard_normal(2) + 1j * rng.standard_normal(2)
            psi = np.kron(spin / np.linalg.norm(spin), psi)
        x = rng.standard_normal((2, 1 << spins))
        out.append((psi + noise * (x[0] + 1j * x[1])).reshape(M, K))
    local = np.zeros((M, K), dtype=complex)
    local[0, 0] = 1.0
    out.append(local)
    return np.stack([x.reshape(-1) for x in out])


@pytest.mark.parametrize("split", [1, 4, 6, 7, 8])
def test_eigenvalues_of_the_plans_own_matrix(gpu, split):
    rng = np.random.default_rng(17 + split)
    K, spins = 1 << split, 2 * split
    M, batches = 1 << (spins - split), 4 if split <= 6 else 1
    states = np.concatenate([states_of(rng, spins, split) for _ in range(batches)])
    W = len(states)
    psi = torch.from_numpy(states).cuda()
    table = np.array([(K, K, M, K, M, K, w << spins, 0, w * K * K) for w in range(W)])
    for prec in PRECISIONS:
        G = torch.zeros(W * K * K, dtype=torch.complex128, device="cuda")
        bg.batched_gemm_grouped(bg.batched_gemm_plan("c128", table, prec, bg.BG_PLAN_HERK), psi,
                                None, G, 1.0, 0.0)
        ent = torch.zeros(W, dtype=torch.float64, device="cuda")
        eig = torch.zeros(W * K, dtype=torch.float64, device="cuda")
        bg.batched_entropy(bg.entropy_plan(W, spins, split, prec=prec), psi, ent, eig)
        bg.check_device_errors()
        lam = np.linalg.eigvalsh(np.swapaxes(host(G).reshape(W, K, K), 1, 2), UPLO="L")
        err = np.abs(host(eig).reshape(W, K) - lam).max(axis=1)
        lim = 8 * K * U * np.abs(lam).max(axis=1)
        mode = "fp64" if prec is None else (prec.slices, prec.beta_bits)
        assert np.all(err <= lim), (mode, (err / lim).max(), np.argmax(err / lim))
