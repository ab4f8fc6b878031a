"""Performance cases of the library: the calls its users make, at the sizes they make them.

A case is a dict of plain values naming a family (``kind``) and its sizes. ``listed()``
gives the fixed ones, ``draw(rng)`` one more of the same ranges. ``prepare`` builds what a
program holds before the call (seeded inputs on the GPU, the plan), ``run`` makes one call
through the public entry points and returns its whole outputs, ``work`` counts the bytes
and flops the operation cannot do without, and ``exact`` computes the same outputs with
plain torch in 64 bits.

Families:
  fixed    batched_gemm_fixed: one shape at a constant stride
  mix      batched_gemm_grouped: square instances, sizes from the 16..512 mix
  ragged   batched_gemm_grouped: rectangular instances of odd sizes, padded leading dimensions
  herk     batched_gemm_grouped with BG_PLAN_HERK: rho = Psi Psi^H for the shapes of spin chains
  chain    chain_step: C_w <- U_t C_w, one pool of unitaries per size
  gate     apply_local_gate on a batch of state vectors
  entropy  batched_entropy with the eigenvalues
  anneal   anneal_step: gate, entropy and Metropolis decision of every walker
"""
import math

import numpy as np
import torch

import paper_2203_09353_gb300 as bg

MIX_SIZES = (16, 32, 64, 128, 256, 512)
MIX_WEIGHTS = (0.30, 0.25, 0.20, 0.15, 0.07, 0.03)


def listed():
    return [
        # the smallest call: a handful of 5-spin operators, where latency is everything
        dict(name="fixed-r64-64x32-fp64", kind="fixed", dtype="r64", m=32, n=32, k=32, batch=64,
             slices=0, alpha=1.0, beta=0.0),
        # 6-spin operators: Hermitian times unitary, one shape, the 9-slice mode
        dict(name="fixed-c128-4096x64-split9", kind="fixed", dtype="c128", m=64, n=64, k=64,
             batch=4096, slices=9, alpha=1.0, beta=0.0),
        # the benchmark's headline: the whole variable-size batch in one 9-slice call
        dict(name="mix-20000-split9", kind="mix", count=20000, values="loguniform", slices=9,
             alpha=1.0, beta=0.5),
        # the same kind of batch in plain FP64, replayed from its captured graph
        dict(name="mix-2000-fp64", kind="mix", count=2000, values="uniform", slices=0,
             alpha=1.0, beta=0.5),
        # rectangular instances of any size up to 300, the quick 3-slice mode
        dict(name="ragged-r64-1500-split3", kind="ragged", dtype="r64", count=1500, edge=300,
             slices=3, alpha=-0.5, beta=0.5),
        # density matrices rho = Psi Psi^H of chains of 13, 15 and 17 spins, 6 slices
        dict(name="herk-13-15-17-split6", kind="herk", each=48, spins="13,15,17", slices=6),
        # the step loop of chained operators: 8-spin walkers beside a few 10-spin ones
        dict(name="chain-240x256-16x1024-split9", kind="chain", n_small=256, walkers_small=240,
             n_large=1024, walkers_large=16, steps=2, slices=9),
        # the local gate of every Monte Carlo step on 1024 chains of 17 spins
        dict(name="gate-1024x17", kind="gate", walkers=1024, spins=17),
        # entanglement entropy of mid-sized chains in plain FP64
        dict(name="entropy-32x15-fp64", kind="entropy", walkers=32, spins=15, slices=0),
        # the paper's run: 21 spins, 16 Monte Carlo procedures on one GPU
        dict(name="entropy-16x21-split9", kind="entropy", walkers=16, spins=21, slices=9),
        # whole annealing steps of 128 procedures, 17 spins
        dict(name="anneal-128x17-split9", kind="anneal", walkers=128, spins=17, slices=9),
        # whole annealing steps at the small end: 4 procedures of 13 spins
        dict(name="anneal-4x13-split9", kind="anneal", walkers=4, spins=13, slices=9),
    ]


# ---- drawing cases --------------------------------------------------------------------------


def _log_int(rng, lo, hi):
    return min(hi, max(lo, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi + 0.49)))))))


def _walkers(rng, spins, lo, hi, cap):
    """Log-spread walkers, within `cap` units of walkers x K^3 (K the Gram order)."""
    most = max(lo, min(hi, cap // (8 ** (spins // 2))))
    return _log_int(rng, lo, most)


def draw(rng):
    kind = rng.choice(("fixed", "mix", "ragged", "herk", "chain", "gate", "entropy", "anneal"))
    if kind == "fixed":
        dtype = rng.choice(("r64", "c128"))
        m, n, k = (_log_int(rng, 8, 64) for _ in range(3))
        if rng.random() < 0.4:
            m = n = k = rng.choice((16, 32, 64))
        slices = rng.choice((0, 3, 6, 9))
        return dict(kind=kind, dtype=dtype, m=m, n=n, k=k,
                    batch=_log_int(rng, 48, 1024 if slices == 0 else 4096), slices=slices,
                    alpha=1.0, beta=rng.choice((0.0, 0.5)))
    if kind == "mix":
        slices = rng.choice((0, 3, 6, 9))
        return dict(kind=kind, count=_log_int(rng, 150, 2000 if slices == 0 else 12000),
                    values=rng.choice(("uniform", "loguniform")), slices=slices, alpha=1.0,
                    beta=0.5)
    if kind == "ragged":
        slices = rng.choice((0, 3, 6, 9))
        dtype = rng.choice(("r64", "c128"))
        return dict(kind=kind, dtype=dtype, count=_log_int(rng, 100, 300 if slices == 0 else 1200),
                    edge=_log_int(rng, 24, 256), slices=slices, alpha=rng.choice((1.0, -0.5)),
                    beta=rng.choice((0.0, 0.5)))
    if kind == "herk":
        spins = sorted(rng.sample(range(9, 18), rng.choice((1, 2, 3))))
        return dict(kind=kind, each=_log_int(rng, 6, 40), spins=",".join(map(str, spins)),
                    slices=rng.choice((0, 6, 9)))
    if kind == "chain":
        large = _log_int(rng, 200, 600)
        return dict(kind=kind, n_small=_log_int(rng, 40, 256), walkers_small=_log_int(rng, 20, 240),
                    n_large=large, walkers_large=_log_int(rng, 2, 16), steps=rng.choice((1, 2, 4)),
                    slices=rng.choice((3, 6, 9)))
    if kind == "gate":
        spins = rng.randint(9, 19)
        return dict(kind=kind, walkers=_log_int(rng, 8, min(1024, 1 << (27 - spins))), spins=spins)
    slices = rng.choice((0, 9, 9, 6))
    spins = rng.randint(8, 17 if slices == 0 else 20)
    cap = (32 if slices == 0 else 512) * (1 << 21)
    if kind == "entropy":
        return dict(kind=kind, walkers=_walkers(rng, spins, 3, 128, cap), spins=spins, slices=slices)
    return dict(kind=kind, walkers=_walkers(rng, min(spins, 18), 3, 128, cap),
                spins=min(spins, 18), slices=slices)


# ---- inputs ---------------------------------------------------------------------------------


def _gen(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(int(seed) * 1000003 + 17)
    return g


def _shape_rng(case):
    """Sizes depend on the case alone: another seed gives other values of the same sizes."""
    return np.random.default_rng(sum(ord(c) * (i + 1) for i, c in enumerate(
        ",".join("%s=%s" % (k, case[k]) for k in sorted(case) if k != "name"))))


def _prec(case):
    s = case.get("slices", 0)
    return bg.precision("split", s) if s else None


def _pairs(case):
    """Real multiply-adds spent per product term: s (s + 1) / 2 plane pairs in the split mode."""
    s = case["slices"]
    return s * (s + 1) // 2 if s else 1


def _uniform(n, g):
    return torch.rand(n, generator=g, device="cuda", dtype=torch.float64).mul_(2.0).sub_(1.0)


def _loguniform(n, g):
    """10^U(-4, 4) with a random sign."""
    x = torch.pow(10.0, torch.rand(n, generator=g, device="cuda", dtype=torch.float64) * 8.0 - 4.0)
    sign = torch.randint(0, 2, (n,), generator=g, device="cuda", dtype=torch.int8)
    return x * (1.0 - 2.0 * sign)


def _cnormal(shape, g):
    return torch.view_as_complex(torch.randn((*shape, 2), generator=g, device="cuda",
                                             dtype=torch.float64))


def _cuniform(n, g):
    return torch.view_as_complex(_uniform(2 * n, g).view(n, 2))


def _haar(n, count, g):
    """`count` Haar unitaries of order n (QR of a complex Gaussian, phases of R's diagonal)."""
    q, r = torch.linalg.qr(_cnormal((count, n, n), g))
    d = torch.diagonal(r, dim1=-2, dim2=-1)
    return q * (d / d.abs()).unsqueeze(-2)


def _phases(shape, g):
    t = torch.rand(shape, generator=g, device="cuda", dtype=torch.float64) * (2.0 * math.pi)
    return torch.polar(torch.ones_like(t), t)


def _gates(walkers, rng):
    z = rng.standard_normal((walkers, 4, 4)) + 1j * rng.standard_normal((walkers, 4, 4))
    q, r = np.linalg.qr(z)
    d = np.diagonal(r, axis1=1, axis2=2)
    return q * (d / np.abs(d))[:, None, :]


def _states(walkers, spins, g):
    s = _cnormal((walkers, 1 << spins), g)
    return s / torch.linalg.vector_norm(s, dim=1, keepdim=True)


def _table(case):
    """Instance table (m, n, k, lda, ldb, ldc, offsets) and the operand lengths."""
    rng = _shape_rng(case)
    if case["kind"] == "mix":
        ns = rng.choice(np.asarray(MIX_SIZES), size=case["count"], p=np.asarray(MIX_WEIGHTS))
        shapes = [(int(x),) * 3 for x in ns]
        pad = np.zeros((len(shapes), 3), dtype=np.int64)
    elif case["kind"] == "ragged":
        e = np.exp(rng.uniform(math.log(5), math.log(case["edge"] + 0.49), (case["count"], 3)))
        shapes = [tuple(int(round(x)) for x in row) for row in e]
        pad = rng.integers(0, 6, (case["count"], 3))
    else:  # herk: Psi of 2^(S - floor(S/2)) x 2^floor(S/2)
        shapes = []
        for s in (int(x) for x in case["spins"].split(",")):
            shapes += [(1 << (s - s // 2), 1 << (s - s // 2), 1 << (s // 2))] * case["each"]
        pad = np.zeros((len(shapes), 3), dtype=np.int64)
    rows, off = [], [0, 0, 0]
    for (m, n, k), p in zip(shapes, pad):
        lda, ldb, ldc = m + int(p[0]), k + int(p[1]), m + int(p[2])
        rows.append((m, n, k, lda, ldb, ldc, *off))
        for i, size in enumerate((lda * k, ldb * n, ldc * n)):
            off[i] = (off[i] + size + 31) // 32 * 32
    return np.array(rows, dtype=np.int64), off


def _inputs(case, seed):
    g = _gen(seed)
    kind = case["kind"]
    if kind == "fixed":
        m, n, k, b = case["m"], case["n"], case["k"], case["batch"]
        if case["dtype"] == "c128":
            A = _cnormal((b, k, m), g)
            if m == k:  # Hermitian operators
                A = 0.5 * (A + A.conj().transpose(1, 2)).resolve_conj()
            B = _cnormal((b, n, k), g) / math.sqrt(2.0 * k)
            C = _cnormal((b, n, m), g)
            return dict(A=A.contiguous(), B=B, C=C)
        return dict(A=_uniform(b * k * m, g).view(b, k, m), B=_uniform(b * n * k, g).view(b, n, k),
                    C=_uniform(b * n * m, g).view(b, n, m))
    if kind in ("mix", "ragged", "herk"):
        table, (la, lb, lc) = _table(case)
        if kind == "herk":
            return dict(table=table, A=_cnormal((la,), g), B=None,
                        C=torch.zeros(lc, device="cuda", dtype=torch.complex128))
        if case.get("dtype", "r64") == "c128":
            return dict(table=table, A=_cuniform(la, g), B=_cuniform(lb, g), C=_cuniform(lc, g))
        fill = _loguniform if case.get("values") == "loguniform" else _uniform
        return dict(table=table, A=fill(la, g), B=fill(lb, g), C=fill(lc, g))
    if kind == "chain":
        pools, states = [], []
        rng = np.random.default_rng(seed)
        idx = []
        base = 0
        for n, walkers, count in ((case["n_small"], case["walkers_small"], 8),
                                  (case["n_large"], case["walkers_large"], 3)):
            U = _haar(n, count, g)
            pools.append(U)
            # unitary start states: pool unitaries between random diagonal phases
            pick = torch.arange(walkers, device="cuda") % count
            states.append(_phases((walkers, n, 1), g) * U[pick] * _phases((walkers, 1, n), g))
            idx.append(base + rng.integers(0, count, (case["steps"], walkers)))
            base += count
        return dict(pools=pools, states=states,
                    idx=torch.from_numpy(np.concatenate(idx, axis=1).astype(np.int32)).cuda())
    states = _states(case["walkers"], case["spins"], g)
    if kind == "entropy":
        return dict(states=states)
    rng = np.random.default_rng(seed)
    gates = _gates(case["walkers"], rng)
    sites = rng.integers(0, case["spins"] - 1, case["walkers"]).astype(np.int32)
    d = dict(states=states, sites=torch.from_numpy(sites).cuda(), gates_host=gates,
             gates=torch.from_numpy(np.ascontiguousarray(gates.transpose(0, 2, 1))).cuda())
    if kind == "anneal":
        d["uniforms"] = torch.from_numpy(rng.random(case["walkers"])).cuda()
    return d


TEMPERATURE = 0.05


def prepare(case, seed):
    d = _inputs(case, seed)
    d["case"] = case
    kind = case["kind"]
    prec = _prec(case)
    if kind == "fixed":
        d["prec"] = prec
    elif kind in ("mix", "ragged", "herk"):
        flags = bg.BG_PLAN_HERK if kind == "herk" else 0
        if kind == "mix" and not case["slices"]:
            flags |= bg.BG_PLAN_CAPTURE_GRAPH
        dtype = "c128" if kind == "herk" else case.get("dtype", "r64")
        d["plan"] = bg.batched_gemm_plan(dtype, d["table"], prec, flags)
    elif kind == "chain":
        wn, woff, pn, poff = [], [], [], []
        off = poff_next = 0
        for U, S in zip(d["pools"], d["states"]):
            n = U.shape[-1]
            for _ in range(U.shape[0]):
                pn.append(n)
                poff.append(poff_next)
                poff_next += n * n
            for _ in range(S.shape[0]):
                wn.append(n)
                woff.append(off)
                off += n * n
        # column-major storage of each matrix
        d["pool"] = torch.cat([U.transpose(1, 2).reshape(-1) for U in d["pools"]])
        d["ping"] = torch.cat([S.transpose(1, 2).reshape(-1) for S in d["states"]])
        d["pong"] = torch.zeros_like(d["ping"])
        d["plan"] = bg.chain_plan("c128", wn, woff, pn, poff, prec)
        del d["states"], d["pools"]
    elif kind == "entropy":
        w, s = case["walkers"], case["spins"]
        d["plan"] = bg.entropy_plan(w, s, prec=prec)
        d["entropy"] = torch.zeros(w, device="cuda", dtype=torch.float64)
        d["eigs"] = torch.zeros((w, 1 << (s // 2)), device="cuda", dtype=torch.float64)
    elif kind == "anneal":
        w, s = case["walkers"], case["spins"]
        start = bg.entropy_plan(w, s, prec=prec)
        d["energy"] = torch.zeros(w, device="cuda", dtype=torch.float64)
        bg.batched_entropy(start, d["states"], d["energy"])
        d["plan"] = bg.anneal_plan(w, s, prec=prec)
        d["accepted"] = torch.zeros(w, device="cuda", dtype=torch.int32)
        torch.cuda.synchronize()
        start.close()
    return d


def run(state):
    d, case = state, state["case"]
    kind = case["kind"]
    if kind == "fixed":
        m, n, k = case["m"], case["n"], case["k"]
        bg.batched_gemm_fixed(case["dtype"], m, n, k, case["alpha"], d["A"], m, m * k, d["B"], k,
                              k * n, case["beta"], d["C"], m, m * n, case["batch"], d["prec"])
        return d["C"]
    if kind in ("mix", "ragged"):
        bg.batched_gemm_grouped(d["plan"], d["A"], d["B"], d["C"], case["alpha"], case["beta"])
        return d["C"]
    if kind == "herk":
        bg.batched_gemm_grouped(d["plan"], d["A"], None, d["C"], 1.0, 0.0)
        return d["C"]
    if kind == "chain":
        bg.chain_step(d["plan"], d["pool"], d["idx"], d["ping"], d["pong"], case["steps"])
        return d["ping"] if case["steps"] % 2 == 0 else d["pong"]
    if kind == "gate":
        bg.apply_local_gate(d["states"], case["spins"], d["sites"], d["gates"])
        return d["states"]
    if kind == "entropy":
        bg.batched_entropy(d["plan"], d["states"], d["entropy"], d["eigs"])
        return d["entropy"], d["eigs"]
    bg.anneal_step(d["plan"], d["states"], d["energy"], d["sites"], d["gates"], d["uniforms"],
                   TEMPERATURE, 1, d["accepted"])
    return d["states"], d["energy"], d["accepted"]


# ---- what a pass cannot do without -------------------------------------------------------------


def _entropy_work(walkers, spins, pairs):
    K, M = 1 << (spins // 2), 1 << (spins - spins // 2)
    # the lower triangle of X X^H, then the Householder reduction of a Hermitian matrix
    return dict(bytes=walkers * (16.0 * K * M + 8.0 * (K + 1)),
                flops=walkers * (pairs * 4.0 * K * K * M + 16.0 / 3.0 * K ** 3))


def work(case):
    kind = case["kind"]
    if kind in ("fixed", "mix", "ragged", "herk"):
        if kind == "fixed":
            t = np.array([[case["m"], case["n"], case["k"]]] * case["batch"], dtype=np.float64)
        else:
            t = _table(case)[0][:, :3].astype(np.float64)
        m, n, k = t[:, 0], t[:, 1], t[:, 2]
        cplx = kind == "herk" or case.get("dtype") == "c128"
        esz, per = (16.0, 8.0) if cplx else (8.0, 2.0)
        if kind == "herk":
            return dict(bytes=float(esz * np.sum(m * k + n * (n + 1) / 2)),
                        flops=float(_pairs(case) * per * np.sum(n * (n + 1) / 2 * k)))
        c = 2.0 if case["beta"] != 0 else 1.0
        return dict(bytes=float(esz * np.sum(m * k + k * n + c * m * n)),
                    flops=float(_pairs(case) * per * np.sum(m * n * k)))
    if kind == "chain":
        b = f = 0.0
        for n, w, count in ((case["n_small"], case["walkers_small"], 8),
                            (case["n_large"], case["walkers_large"], 3)):
            b += 16.0 * n * n * (2 * w + count)
            f += 8.0 * float(n) ** 3 * w * case["steps"]
        return dict(bytes=b, flops=f * _pairs(case))
    amps = float(case["walkers"]) * (1 << case["spins"])
    if kind == "gate":
        return dict(bytes=32.0 * amps, flops=32.0 * amps)
    w = _entropy_work(case["walkers"], case["spins"], _pairs(case))
    if kind == "entropy":
        return w
    # the state read, the accepted proposals written; gate flops
    return dict(bytes=w["bytes"] + 16.0 * amps, flops=w["flops"] + 32.0 * amps)


# ---- 64-bit results ------------------------------------------------------------------------------


def _apply_gates(states, sites, gates):
    out = states.clone()
    for w in range(states.shape[0]):
        j = int(sites[w])
        v = states[w].view(-1, 4, 1 << j)  # index b_j + 2 b_{j+1} in the middle
        u = torch.from_numpy(gates[w]).to(states.device)
        out[w] = torch.einsum("ac,hcl->hal", u, v).reshape(-1)
    return out


def _spectra(states, spins):
    """Ascending eigenvalues of the Gram matrix across the cut, and the entropies."""
    K = 1 << (spins // 2)
    X = states.view(states.shape[0], -1, K).transpose(1, 2)  # K x M
    lam = torch.stack([torch.linalg.eigvalsh(x @ x.conj().T) for x in X])
    p = lam / lam.sum(dim=1, keepdim=True)
    pos = p > 0
    logs = torch.where(pos, torch.log(torch.where(pos, p, torch.ones_like(p))),
                       torch.zeros_like(p))
    return lam, -(p.clamp_min(0.0) * logs).sum(dim=1)


def exact(case, seed):
    d = _inputs(case, seed)
    kind = case["kind"]
    if kind == "fixed":
        # stored [k, m] and [n, k]: the transposes of the column-major matrices
        C = case["alpha"] * torch.bmm(d["B"], d["A"])
        return C + case["beta"] * d["C"] if case["beta"] != 0 else C
    if kind in ("mix", "ragged", "herk"):
        C = d["C"]
        for m, n, k, lda, ldb, ldc, ao, bo, co in d["table"].tolist():
            a = d["A"][ao:ao + lda * k].view(k, lda)[:, :m]
            c = C[co:co + ldc * n].view(n, ldc)[:, :m]
            if kind == "herk":  # c[j, i] = sum_p a[p, i] conj(a[p, j]), i >= j
                c.copy_(torch.triu(a.conj().T @ a))
                c.diagonal().imag.zero_()
            else:
                b = d["B"][bo:bo + ldb * n].view(n, ldb)[:, :k]
                c.copy_(case["alpha"] * (b @ a) + case["beta"] * c)
        return C
    if kind == "chain":
        out, base = [], 0
        col = 0
        for U, S in zip(d["pools"], d["states"]):
            ids = d["idx"][:, col:col + S.shape[0]].long() - base
            for t in range(case["steps"]):
                S = torch.bmm(U[ids[t]], S)
            out.append(S.transpose(1, 2).reshape(-1))
            base += U.shape[0]
            col += ids.shape[1]
        return torch.cat(out)
    if kind == "gate":
        return _apply_gates(d["states"], d["sites"].cpu(), d["gates_host"])
    if kind == "entropy":
        lam, ent = _spectra(d["states"], case["spins"])
        return ent, lam
    cur = d["states"]
    prop = _apply_gates(cur, d["sites"].cpu(), d["gates_host"])
    e_cur, e_new = _spectra(cur, case["spins"])[1], _spectra(prop, case["spins"])[1]
    delta = e_new - e_cur
    acc = (delta <= 0) | (d["uniforms"] < torch.exp(-delta / TEMPERATURE))
    return (torch.where(acc.unsqueeze(1), prop, cur), torch.where(acc, e_new, e_cur),
            acc.to(torch.int32))
