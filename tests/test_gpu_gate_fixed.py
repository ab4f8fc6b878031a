"""The fixed-point route of apply_local_gate at its edges: which gates and
groups take it, and what the two routes give for values far apart, at the ends
of the exponent range, zeros, infinities and NaN.

Tolerance. A group's fixed-point result is off by at most 2^-58 of the
group's largest component times the gate's row sum (59-bit amplitudes and
gate entries, cut cross sums) plus one rounding to FP64; the FP64 chain of
the oracle by at most 8 x 2^-53 of the same product. Their difference is
below 2^-49 max|psi| sum|U| for every component of a group.
"""
import numpy as np
import pytest
import torch

import oracle
import paper_2203_09353_gb300 as bg

from gpu_util import host

pytestmark = pytest.mark.gpu


def haar4(rng):
    z = rng.standard_normal((4, 4)) + 1j * rng.standard_normal((4, 4))
    q, r = np.linalg.qr(z)
    return q * (np.diag(r) / np.abs(np.diag(r)))


def run(psi, S, sites, U):
    st = torch.from_numpy(psi.reshape(-1).copy()).cuda()
    s = torch.from_numpy(np.asarray(sites, dtype=np.int32)).cuda()
    g = torch.from_numpy(np.ascontiguousarray(np.asarray(U).transpose(0, 2, 1)).ravel()).cuda()
    bg.apply_local_gate(st, S, s, g)
    bg.check_device_errors()
    return host(st).reshape(psi.shape)


def check(got, psi, S, sites, U):
    ref = oracle.two_site_gate(psi, S, sites, U)
    for w in range(psi.shape[0]):
        sh = (-1, 4, 1 << int(sites[w]))
        big = np.abs(psi[w]).reshape(sh).max(axis=1, keepdims=True)
        row = np.abs(U[w]).sum(axis=1)[None, :, None]
        assert np.all(np.abs((got[w] - ref[w]).reshape(sh)) <= 2.0 ** -49 * big * row), w


@pytest.mark.parametrize("S,W", [(2, 5), (3, 1), (9, 700), (13, 3), (17, 2)])
def test_sizes(gpu, S, W):
    rng = np.random.default_rng(600 + S)
    psi = rng.standard_normal((W, 1 << S)) + 1j * rng.standard_normal((W, 1 << S))
    sites = rng.integers(0, S - 1, W).astype(np.int32)
    U = np.stack([haar4(rng) for _ in range(W)])
    check(run(psi, S, sites, U), psi, S, sites, U)


def test_spread_and_extreme_amplitudes(gpu):
    """Amplitudes over forty decades inside a group, whole groups near the ends
    of the exponent range (both routes), zero groups, zeros beside values."""
    rng = np.random.default_rng(610)
    S, W = 8, 6
    psi = rng.standard_normal((W, 1 << S)) + 1j * rng.standard_normal((W, 1 << S))
    psi[0] *= 10.0 ** rng.uniform(-40, 0, 1 << S)
    psi[1] *= 10.0 ** np.repeat(rng.uniform(-290, 290, 1 << (S - 2)), 4)
    psi[2, ::3] = 0.0
    psi[3, : 1 << (S - 1)] = 0.0
    psi[4] *= 2.0 ** np.repeat(rng.integers(-725, -715, 1 << (S - 2)).astype(float), 4)
    psi[5] = psi[5].real
    sites = np.zeros(W, dtype=np.int32)
    U = np.stack([haar4(rng) for _ in range(W)])
    got = run(psi, S, sites, U)
    check(got, psi, S, sites, U)
    assert np.all(got[3, : 1 << (S - 1)] == 0.0)


def test_gate_entry_ratios(gpu):
    """Gates with entries on both sides of the ratio that the fixed-point route
    takes, scaled gates, gates with zeros."""
    rng = np.random.default_rng(620)
    S = 6
    U = []
    for e in (4, 5, 6, 7, 8, 30):
        u = haar4(rng)
        u[1, 2] *= 2.0 ** -e / abs(u[1, 2])
        U.append(u)
    U += [haar4(rng) * 2.0 ** 100, haar4(rng) * 2.0 ** -130, haar4(rng).real + 0j,
          np.kron(haar4(rng)[:2, :2], np.eye(2))]
    U = np.stack(U)
    W = len(U)
    psi = rng.standard_normal((W, 1 << S)) + 1j * rng.standard_normal((W, 1 << S))
    psi[:, ::4] *= 1e-9  # rows whose large terms meet the small entries
    sites = rng.integers(0, S - 1, W).astype(np.int32)
    check(run(psi, S, sites, U), psi, S, sites, U)


def test_non_finite(gpu):
    """A NaN or infinity spreads over its own group of four and no further."""
    rng = np.random.default_rng(630)
    S = 6
    psi = rng.standard_normal((3, 1 << S)) + 1j * rng.standard_normal((3, 1 << S))
    clean = psi.copy()
    psi[0, 5] = np.nan
    psi[1, 9] = np.inf
    U = np.stack([haar4(rng) for _ in range(3)])
    U[2, 0, 0] = np.nan
    got, ref = run(psi, S, [0, 0, 0], U), run(clean, S, [0, 0, 0], np.stack([U[0], U[1], U[0]]))
    assert not np.isfinite(got[0, 4:8]).any() and not np.isfinite(got[1, 8:12]).any()
    keep0 = np.r_[0:4, 8:1 << S]
    assert np.array_equal(got[0, keep0], ref[0, keep0])
    assert np.isnan(got[2, 0::4]).all() and np.isfinite(got[2, 1::4]).all()
