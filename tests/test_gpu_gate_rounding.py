"""The error of apply_local_gate's fixed-point route against an exact product
(double-double), in its own units u = 2^(E + EU - 58), where a group's largest
component lies in [2^(E-1), 2^E) and the gate's in [2^(EU-1), 2^EU).

Tolerances, each followed by one rounding to FP64 (half an ulp):
  - at most 13 u: operands cut to 59 bits are 1 (psi) and 1/2 (U) of 2^-59 off,
    0.75 u for each of the 8 real products of an output; the product of two low
    limbs, below u / 4 each, is dropped 8 times (re), or 4 times with both
    factors doubled and 8 times (im): 2 and 6 u; one rounding, half a unit:
    8.5 and 12.5 u.
  - rms: the same terms as independent errors. Cuts of psi are uniform in [0, 1)
    with the amplitude's sign, 1/3 each, times |U|^2, which a row sums to 1:
    1/12 u^2; those of U 1/12 each, at most 8 times 1/4: 1/6; dropped products
    uniform factors, 1/144 each, 8 (re) or 24 (im) of them: 1/18 and 1/6;
    rounding 1/12. Together 0.39 and 0.5 u^2: below 0.75 u, where the result
    is small enough that its own rounding adds less than u / 8.
  - mean: zero. Of some 5000 such results its spread is 0.75 / 70 = 0.011 u.
"""
import numpy as np
import pytest
import torch

import oracle
import paper_2203_09353_gb300 as bg

from gpu_util import host

pytestmark = pytest.mark.gpu


def two_sum(a, b):
    s = a + b
    t = s - a
    return s, (a - (s - t)) + (b - t)


def two_prod(a, b):
    p = a * b
    ta, tb = a * 134217729.0, b * 134217729.0
    ah, bh = ta - (ta - a), tb - (tb - b)
    al, bl = a - ah, b - bh
    return p, ((ah * bh - p) + ah * bl + al * bh) + al * bl


def exact_error(got, terms):
    """got - sum of the products, to double-double precision."""
    hi, lo = got, np.zeros_like(got)
    for a, b in terms:
        p, q = two_prod(-a, b)
        hi, e = two_sum(hi, p)
        lo = lo + (e + q)
    return hi + lo


def haar4(rng):
    z = rng.standard_normal((4, 4)) + 1j * rng.standard_normal((4, 4))
    q, r = np.linalg.qr(z)
    return q * (np.diag(r) / np.abs(np.diag(r)))


def fixed_route_gates(rng, count):
    """Haar gates that the fixed-point route takes (entries within 2^6 of each other)."""
    out = []
    while len(out) < count:
        u = haar4(rng)
        m = np.maximum(np.abs(u.real), np.abs(u.imag))
        if m.min() >= m.max() * 2.0 ** -5:
            out.append(u)
    return np.stack(out)


@pytest.mark.parametrize("spread", ["random", "one large"])
def test_error_in_units(gpu, spread):
    S, W = 15, 64
    rng = np.random.default_rng(640)
    psi = rng.standard_normal((W, 1 << S)) + 1j * rng.standard_normal((W, 1 << S))
    if spread == "one large":
        psi.reshape(W, -1, 4)[:, :, 1:] *= 1e-3
    U = fixed_route_gates(rng, W)
    sites = np.zeros(W, dtype=np.int32)
    st = torch.from_numpy(psi.reshape(-1).copy()).cuda()
    g = torch.from_numpy(np.ascontiguousarray(U.transpose(0, 2, 1)).ravel()).cuda()
    bg.apply_local_gate(st, S, torch.from_numpy(sites).cuda(), g)
    bg.check_device_errors()
    got = host(st).reshape(W, -1, 4)
    chain = oracle.two_site_gate(psi, S, sites, U).reshape(W, -1, 4)
    v = psi.reshape(W, -1, 4)

    def top(z, axes):
        return np.frexp(np.maximum(np.abs(z.real), np.abs(z.imag)).max(axis=axes, keepdims=True))[1]

    unit = np.ldexp(1.0, top(v, 2) + top(U, (1, 2)) - 58)
    vals, errs, chains = [], [], []
    for a in range(4):
        re, im = [], []
        for c in range(4):
            x, y = U[:, a, c].real[:, None], U[:, a, c].imag[:, None]
            p, q = v[:, :, c].real, v[:, :, c].imag
            re += [(x, p), (-y, q)]
            im += [(x, q), (y, p)]
        for part, terms in (("real", re), ("imag", im)):
            z = getattr(got[:, :, a], part)
            vals.append(z)
            errs.append(exact_error(z, terms) / unit[:, :, 0])
            chains.append(exact_error(getattr(chain[:, :, a], part), terms) / unit[:, :, 0])
    vals, errs, chains = (np.stack(x) for x in (vals, errs, chains))
    half_ulp = np.spacing(np.abs(vals)) / 2 / unit[None, :, :, 0]
    assert np.all(np.abs(errs) <= 13.0 + half_ulp)
    assert np.sqrt(np.mean(errs ** 2)) <= np.sqrt(np.mean(chains ** 2))
    small = errs[half_ulp <= 0.125]
    assert small.size > 2000
    assert np.sqrt(np.mean(small ** 2)) <= 0.75 + 0.125
    assert abs(np.mean(small)) <= 0.1
