"""The calls whose time matters to a program that uses this library, at the sizes it uses.

Every case is one call sequence through the public entry points (``Context``, ``ExchangeEnergy``,
``build_batch``, ``term_noalloc``):

  op "scf"       one step of a self-consistent loop: the new density matrix is set (device data), the
                 exchange matrix is built, its keys and values are taken (values on the device).  The
                 context, with C and V set and one build behind it, is what such a loop keeps.
  op "geometry"  one step of a relaxation or of molecular dynamics: new C, V and D from page-locked
                 host memory into the kept context, a build, and every block read back to the host.
  op "grad"      energy and gradients with respect to C and V through the autograd wrapper.
  op "batch"     many small independent cells built together, each with its own threshold.
  op "density"   real-space density matrix from eigenvectors (host arrays in and out).
  op "sigma_k"   the built exchange matrix at k points (host array out).
  op "term"      one exchange term without device allocation.

Cells are diamond-cubic (one element), rocksalt-like (two elements) or a small odd cluster; block
values follow the decay with distance of numerical atomic orbitals: C ~ exp(-d/2), V ~ erfc(mu d)/d,
D ~ exp(-d/3) for an insulator or (1 + d/3)^-2 for a metal.  A block's largest value is set by its
distance alone, so the screen keeps the same terms, and the exchange matrix has the same blocks, for
every draw of the values.
"""
import itertools
import math

import numpy as np
import torch

from paper_2009_12505_gb300 import hfx

SI = {"lattice": "diamond", "ncell": 1, "nao": 13, "nabf": 60, "nao2": 13, "nabf2": 60,
      "cut_C": 16.0, "cut_V": 20.0, "cut_D": 16.0, "mu": 0.11, "metal": False,
      "theta": 1e-6, "prec": "ozaki", "nslices": 6, "eri": -1.0}


def _case(name, op, **kw):
    return {**SI, **kw, "op": op, "name": name}


def listed():
    return [
        # one exchange term for a caller that may not allocate: the smallest call
        _case("term", "term", nao2=27, nabf2=90),
        # three odd-sized atoms in FP64: the smallest whole build, where launches and waits count
        _case("cluster_fp64", "scf", lattice="cluster", nao=4, nabf=5, nao2=2, nabf2=3, cut_C=3.2,
              cut_V=4.2, cut_D=3.0, theta=1e-2, prec="fp64", nslices=0),
        # SCF step of the conventional 8-atom cell, at the cutoffs and threshold of the benchmark
        _case("si8_scf", "scf"),
        # SCF step of the 2x2x2 supercell: the largest
        _case("si64_scf", "scf", ncell=2),
        # SCF step of a two-element cell with uneven 13/60 and 27/90 blocks, shorter cutoffs
        _case("ab8_scf", "scf", lattice="rocksalt", nao2=27, nabf2=90, cut_C=9.0, cut_V=12.0,
              cut_D=9.0),
        # a metal (slow decay of D) with both screens on, as both are used together, taken to k points
        _case("metal8_eri_scf", "scf", cut_D=24.0, metal=True, eri=1e-3, nk=2),
        # the 8-atom cell in FP64, to check a split-precision run against
        _case("si8_fp64", "scf", cut_C=12.0, cut_V=16.0, cut_D=12.0, prec="fp64", nslices=0),
        # a relaxation step: everything set again from the host, the result read back
        _case("si8_geometry", "geometry"),
        # forces or basis optimisation: energy, dE/dC and dE/dV of a short-range cell
        _case("si8_grad", "grad", cut_C=8.0, cut_V=10.0, cut_D=8.0),
        # a set of small cells of one and two elements, thresholds 1e-5 .. 1e-7
        _case("batch6", "batch", ncells=6, nao2=27, nabf2=90, cut_C=7.0, cut_V=9.0, cut_D=7.0),
        # density matrix of the 64-atom cell from a 2x2x2 k grid
        _case("si64_density", "density", ncell=2, nk=2),
        # exchange matrix of the 64-atom cell (short cutoffs) on a 2x2x2 k grid
        _case("si64_sigma_k", "sigma_k", ncell=2, nk=2, cut_C=8.0, cut_V=10.0, cut_D=8.0),
    ]


# Largest canonical flop count of a drawn case: below that of the largest listed case for the
# split builds, and what FP64 units do in about the same time for the others.
MOST_FLOPS = {"split": 12e12, "fp64": 0.5e12, "grad": 0.15e12, "batch": 2e12}


def _log(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def draw(rng):
    op = rng.choice(["scf"] * 7 + ["geometry"] * 2 + ["grad", "batch", "density", "sigma_k"] +
                    ["term"] * 2)
    c = dict(SI, op=op)
    if op == "term":
        while True:
            c["nao"], c["nao2"] = round(_log(rng, 4, 32)), round(_log(rng, 4, 32))
            c["nabf"], c["nabf2"] = round(_log(rng, 20, 200)), round(_log(rng, 20, 200))
            if c["nabf"] * c["nao2"] * max(c["nao"], c["nao2"]) <= 131072:
                return c
    c["nao"], c["nabf"] = round(_log(rng, 4, 30)), round(_log(rng, 20, 100))
    c["nao2"], c["nabf2"] = c["nao"], c["nabf"]
    c["lattice"] = "diamond"
    if rng.random() < 0.35:
        c["lattice"] = "rocksalt"
        c["nao2"], c["nabf2"] = round(_log(rng, 4, 30)), round(_log(rng, 20, 100))
    if op == "density":
        c["ncell"], c["nk"] = rng.choice([1, 2]), rng.choice([1, 2, 3])
        c["nao"], c["nao2"] = min(c["nao"], 14), min(c["nao2"], 14)
        c["cut_D"] = rng.uniform(8.0, 18.0)
        return c
    most = MOST_FLOPS["split"]
    c["cut_C"], c["theta"] = rng.uniform(7.0, 16.0), _log(rng, 1e-7, 1e-4)
    if op == "scf":
        c["ncell"] = rng.choice([1, 1, 1, 2])
        c["nslices"] = rng.choice([6, 6, 6, 5, 4])
        if rng.random() < 0.2:
            c["prec"], c["nslices"], most = "fp64", 0, MOST_FLOPS["fp64"]
        if rng.random() < 0.2:
            c["eri"], c["nk"] = _log(rng, 1e-4, 1e-2), rng.choice([1, 2])
        c["metal"] = rng.random() < 0.2
    elif op == "grad":
        most, c["cut_C"] = MOST_FLOPS["grad"], rng.uniform(5.0, 9.0)
    elif op == "batch":
        most, c["cut_C"] = MOST_FLOPS["batch"], rng.uniform(6.0, 8.0)
        c["ncells"] = rng.randint(2, 10)
    elif op == "sigma_k":
        c["cut_C"], c["ncell"], c["nk"] = rng.uniform(6.0, 9.0), rng.choice([1, 2]), rng.choice([1, 2, 3])
        c["nao"], c["nao2"] = min(c["nao"], 14), min(c["nao2"], 14)
    while True:
        c["cut_V"] = 1.25 * c["cut_C"]
        c["cut_D"] = c["cut_C"] * (1.5 if c["metal"] else 1.0)
        if work(c)["flops"] <= most or c["cut_C"] < 5.0:
            return c
        c["cut_C"] *= 0.93


# ------------------------------------------------------------------------------------ the cell

def _system(c):
    """(grid spacing, period in steps, grid coordinates, nao, nabf) of a cubic cell."""
    if c["lattice"] == "cluster":
        grid = np.array([[0, 0, 0], [2, 1, 0], [1, 3, 2]])
        nao = [c["nao"], c["nao2"], (c["nao"] + c["nao2"]) // 2]
        nabf = [c["nabf"], c["nabf2"], (c["nabf"] + c["nabf2"]) // 2]
        return 1.0, 5, grid, np.array(nao, np.int32), np.array(nabf, np.int32)
    if c["lattice"] == "diamond":
        unit, step = 10.26 / 4.0, 4
        fcc = [(0, 0, 0), (0, 2, 2), (2, 0, 2), (2, 2, 0)]
        basis = fcc + [(x + 1, y + 1, z + 1) for x, y, z in fcc]
    else:
        unit, step = 4.0, 2
        basis = list(itertools.product((0, 1), repeat=3))
    n = c["ncell"]
    grid = np.array([[b[k] + step * t[k] for k in range(3)]
                     for t in itertools.product(range(n), repeat=3) for b in basis])
    second = grid.sum(1) % 2 == 1 if c["lattice"] == "rocksalt" else np.zeros(len(grid), bool)
    return (unit, step * n, grid, np.where(second, c["nao2"], c["nao"]).astype(np.int32),
            np.where(second, c["nabf2"], c["nabf"]).astype(np.int32))


def _pairs(sys_, cut):
    """Keys (i, j, n) of every pair within cut, in key order, and their distances."""
    unit, period, grid = sys_[:3]
    reach = int(math.ceil(cut / (unit * period))) + 1
    shifts = np.array(list(itertools.product(range(-reach, reach + 1), repeat=3)))
    dv = (grid[None, :, None, :] - grid[:, None, None, :]) + shifts * period
    m = (dv * dv).sum(-1)
    i, j, s = np.nonzero(m * (unit * unit) <= cut * cut)
    keys = np.concatenate([np.stack([i, j], 1), shifts[s]], 1).astype(np.int32)
    return keys, np.sqrt(m[i, j, s]) * unit


def _code(k):
    k = k.astype(np.int64)
    return (((k[:, 0] << 20 | k[:, 1]) << 8 | k[:, 2] + 128) << 8 | k[:, 3] + 128) << 8 | k[:, 4] + 128


# Largest value of a block, in units of the decay: that of as many normal draws.
BIG = {"C": 3.9, "V": 3.5, "D": 2.8}


def _decay(c, which, d):
    if which == "C":
        return np.exp(-d / 2.0)
    if which == "V":
        return np.array([math.erfc(c["mu"] * x) for x in d]) / np.maximum(d, 1.0)
    return 0.1 * ((1.0 + d / 3.0) ** -2.0 if c["metal"] else np.exp(-d / 3.0))


class _Blocks:
    """One packed block set: keys and offsets on the host, values on the device."""

    def __init__(self, keys, data, offs):
        self.keys, self.data, self.offs = keys, data, offs


def _blocks(c, sys_, which, seed):
    nao, nabf = sys_[3].astype(np.int64), sys_[4].astype(np.int64)
    keys, d = _pairs(sys_, c["cut_" + which])
    i, j = keys[:, 0], keys[:, 1]
    rows = {"C": nabf[i] * nao[i], "V": nabf[i], "D": nao[i]}[which]
    cols = nabf[j] if which == "V" else nao[j]
    offs = np.concatenate([[0], np.cumsum(rows * cols)])
    gen = torch.Generator("cuda").manual_seed(4 * int(seed) + "CVD".index(which))
    out = torch.empty(int(offs[-1]), dtype=torch.float64, device="cuda")
    site = (i == j) & (keys[:, 2:] == 0).all(1)
    mirror = None
    use = np.ones(len(keys), bool)
    if which != "C":  # V(b, a, -n) = V(a, b, n)^T, and D alike
        code = _code(keys)
        back = np.concatenate([keys[:, 1::-1], -keys[:, 2:]], 1)
        mirror = np.searchsorted(code, _code(back))
        use = mirror >= np.arange(len(keys))
    scale = _decay(c, which, d)
    at = lambda e, n: torch.from_numpy(offs[e]).cuda()[:, None] + torch.arange(n, device="cuda")  # noqa: E731
    for r, q in sorted(set(zip(rows.tolist(), cols.tolist()))):
        e = np.nonzero(use & (rows == r) & (cols == q))[0]
        if not len(e):
            continue
        x = torch.randn(len(e), r, q, dtype=torch.float64, device="cuda", generator=gen)
        s = torch.from_numpy(np.nonzero(site[e])[0]).cuda()
        on = x[s]
        if len(s) and which == "C":
            on = on.view(len(s), -1, q, q)
            on = (on + on.transpose(-1, -2)).reshape(len(s), r, q)
        elif len(s) and which == "V":
            on = on @ on.transpose(-1, -2) / r
            on = 0.5 * (on + on.transpose(-1, -2)) + torch.eye(r, dtype=torch.float64, device="cuda")
        elif len(s):
            on = on + on.transpose(-1, -2)
        x[s] = on
        x *= torch.from_numpy(scale[e]).cuda()[:, None, None] * BIG[which] / x.abs().amax((1, 2), True)
        if len(e) == len(keys):
            out = x.reshape(-1)
            break
        out[at(e, r * q)] = x.reshape(len(e), -1)
        if mirror is not None:
            out[at(mirror[e], r * q)] = x.transpose(-1, -2).reshape(len(e), -1)
    return _Blocks(keys, out, offs)


def _inputs(c, seed):
    sys_ = _system(c)
    return sys_, {k: _blocks(c, sys_, k, seed) for k in "CVD"}


def _context(sys_):
    return hfx.Context(sys_[3], sys_[4], stream=torch.cuda.current_stream().cuda_stream)


def _cells(c):
    """The cells of a batch: diamond and rocksalt-like in turn, thresholds theta x 10, 1, 0.1."""
    return [dict(c, lattice=("diamond", "rocksalt")[q % 2], ncell=1,
                 theta=c["theta"] * (10.0, 1.0, 0.1)[q % 3]) for q in range(c["ncells"])]


def _kgrid(n):
    t = (np.arange(n) + 0.5) / n - 0.5
    return np.array(list(itertools.product(t, repeat=3)))


def _orbitals(c, sys_, seed):
    """Eigenvector coefficients with c(-k) = conj c(k), and occupations: 1.25 x 2 bands an atom."""
    nb, nbands = int(sys_[3].sum()), min(int(sys_[3].sum()), math.ceil(2.5 * len(sys_[3])))
    kf = _kgrid(c["nk"])
    gen = torch.Generator("cuda").manual_seed(4 * int(seed) + 3)
    z = torch.randn(len(kf), nb, nbands, 2, dtype=torch.float64, device="cuda", generator=gen)
    occ = 2.0 * torch.sigmoid(torch.linspace(8.0, -3.0, nbands, dtype=torch.float64, device="cuda")
                              + torch.randn(len(kf), 1, dtype=torch.float64, device="cuda", generator=gen))
    coef = torch.view_as_complex(z / math.sqrt(2.0 * nb))
    half = (len(kf) + 1) // 2  # the grid's second half is the negative of the first, reversed
    for q in range(half, len(kf)):
        coef[q] = coef[len(kf) - 1 - q].conj()
        occ[q] = occ[len(kf) - 1 - q]
    if len(kf) % 2:
        coef[half - 1].imag.zero_()
    return kf, coef.cpu().numpy(), occ.cpu().numpy()


def prepare(case, seed):
    c, op = case, case["op"]
    if op == "term":
        gen = torch.Generator("cuda").manual_seed(int(seed))
        r = lambda *s: torch.randn(*s, dtype=torch.float64, device="cuda", generator=gen)  # noqa: E731
        return {"case": c, "cA": r(c["nabf"], c["nao"], c["nao"]), "V": r(c["nabf"], c["nabf2"]),
                "cB": r(c["nabf2"], c["nao2"], c["nao2"]), "D": 0.1 * r(c["nao"], c["nao2"]),
                "out": torch.empty(c["nao"], c["nao2"], dtype=torch.float64, device="cuda"),
                "stream": torch.cuda.current_stream().cuda_stream}
    if op == "density":
        sys_ = _system(c)
        kf, coef, occ = _orbitals(c, sys_, seed)
        return {"case": c, "ctx": _context(sys_), "kf": kf, "coef": coef, "occ": occ,
                "keys": _pairs(sys_, c["cut_D"])[0]}
    if op == "batch":
        cells = []
        for q, cell in enumerate(_cells(c)):
            sys_, b = _inputs(cell, 100 * int(seed) + q)
            ctx = _context(sys_)
            for k in "CVD":
                ctx.set_blocks(k, b[k], on_device=True)
            cells.append((ctx, b["D"], cell["theta"]))
        return {"case": c, "cells": cells}
    sys_, b = _inputs(c, seed)
    ctx = _context(sys_)
    old = {"D": _blocks(c, sys_, "D", int(seed) + 1000003)}
    if op == "geometry":
        old |= {k: _blocks(c, sys_, k, int(seed) + 1000003) for k in "CV"}
    if c["eri"] >= 0.0:
        ctx.set_eri_screen(c["eri"])
    for k in "CVD":
        ctx.set_blocks(k, b[k] if op in ("grad", "sigma_k") else old.get(k, b[k]), on_device=True)
    ctx.build(c["theta"], c["prec"], c["nslices"])  # the step before this one
    s = {"case": c, "ctx": ctx}
    if op == "geometry":
        s["pinned"] = {k: b[k].data.cpu().pin_memory() for k in "CVD"}
        s["blocks"] = {k: _Blocks(b[k].keys, s["pinned"][k].numpy(), b[k].offs) for k in "CVD"}
    elif op == "grad":
        s |= {k: b[k].data for k in "CVD"}
        s["C"].requires_grad_(True)
        s["V"].requires_grad_(True)
    elif op == "sigma_k":
        s["kf"] = _kgrid(c["nk"])
    else:
        s["D"], s["kf"] = b["D"], _kgrid(c["nk"]) if c["eri"] >= 0.0 else None
    return s


def run(state):
    c, op = state["case"], state["case"]["op"]
    if op == "term":
        return hfx.term_noalloc(state["cA"], state["V"], state["cB"], state["D"], state["out"],
                                state["stream"])
    if op == "batch":
        for ctx, D, _ in state["cells"]:
            ctx.set_blocks("D", D, on_device=True)
        ctxs = [x[0] for x in state["cells"]]
        ex = hfx.build_batch(ctxs, [x[2] for x in state["cells"]], c["prec"], c["nslices"])
        return {"ex": ex, "sigma": [_sigma(ctx) for ctx in ctxs]}
    ctx = state["ctx"]
    if op == "density":
        # the largest imaginary part is rounding noise for such k sets: not an output
        return ctx.density_from_eigvecs(state["kf"], state["coef"], state["occ"], state["keys"])[0]
    if op == "sigma_k":
        return ctx.sigma_k(state["kf"])
    if op == "grad":
        e = hfx.ExchangeEnergy.apply(ctx, c["theta"], c["prec"], c["nslices"], state["C"],
                                     state["V"], state["D"])
        dC, dV = torch.autograd.grad(e, (state["C"], state["V"]))
        return {"ex": e.detach(), "dC": dC, "dV": dV}
    if op == "geometry":
        for k in "CVD":
            ctx.set_blocks(k, state["blocks"][k])
        ex = ctx.build(c["theta"], c["prec"], c["nslices"])
        return {"ex": ex, "keys": ctx.keys(), "sigma": ctx.sigma()}
    ctx.set_blocks("D", state["D"], on_device=True)
    ex = ctx.build(c["theta"], c["prec"], c["nslices"])
    if state["kf"] is not None:  # the ERI screen depends on the values: which blocks remain too
        return {"ex": ex, "sigma_k": ctx.sigma_k(state["kf"])}
    return {"ex": ex, "keys": ctx.keys(), "sigma": _sigma(ctx)}


def _sigma(ctx):
    out = torch.empty(int(ctx.offsets()[-1]), dtype=torch.float64, device="cuda")
    return ctx.sigma(out, on_device=True)


# ------------------------------------------------------------------------------------ the work

def _counts(c, most_b=48):
    """Canonical flops (Algorithm 3: Y once per active (A, B, G), two stages per surviving term)
    from the blocks' largest values, over one atom A of each element and a sample of its B."""
    sys_ = _system(c)
    unit, period, grid, nao, nabf = sys_
    L = unit * period
    pos = grid * unit
    lists = {k: _pairs(sys_, c["cut_" + k]) for k in "CV"}
    val = {k: BIG[k] * _decay(c, k, lists[k][1]) for k in "CV"}
    total = 0.0
    kinds = sorted(set(zip(nao.tolist(), nabf.tolist())))
    for kind in kinds:
        same = (nao == kind[0]) & (nabf == kind[1])
        a = int(np.nonzero(same)[0][0])
        weight = float(same.sum())
        kv, dv = lists["V"]
        mine = np.nonzero(kv[:, 0] == a)[0]
        mine = mine[np.argsort(dv[mine], kind="stable")]
        stride = max(1, len(mine) // most_b)
        kc = lists["C"][0]
        fi = np.nonzero(kc[:, 0] == a)[0]
        pf = pos[kc[fi, 1]] + kc[fi, 2:] * L
        for e in mine[stride // 2::stride]:
            b = int(kv[e, 1])
            gi = np.nonzero(kc[:, 0] == b)[0]
            pb = pos[b] + kv[e, 2:] * L
            pg = pos[kc[gi, 1]] + (kc[gi, 2:] + kv[e, 2:]) * L
            dist = lambda x, y: np.sqrt(((x - y) ** 2).sum(-1))  # noqa: E731

            def live(d):
                return np.where(d <= c["cut_D"] + 1e-9, BIG["D"] * _decay(c, "D", d), 0.0)
            cc = val["C"][fi][:, None] * val["C"][gi][None, :] * val["V"][e]
            nf, ng = nao[kc[fi, 1]].astype(float)[:, None], nao[kc[gi, 1]].astype(float)[None, :]
            na, nb, p = float(nao[a]), float(nao[b]), float(nabf[a])
            away_f = (dist(pf, pos[a]) > 1e-9)[:, None]
            away_g = (dist(pg, pb) > 1e-9)[None, :]
            th = c["theta"]
            m1 = cc * live(dist(pf[:, None], pg[None])) > th
            m2 = (cc * live(dist(pf, pb))[:, None] > th) & away_g
            m3 = (cc * live(dist(pg, pos[a]))[None, :] > th) & away_f
            m4 = (cc * live(np.array(dist(pos[a], pb))) > th) & away_f & away_g
            fl = (m1 * (nb * nf * (ng + na)) + m2 * (nf * ng * (nb + na)) +
                  m3 * (na * nb * (ng + nf)) + m4 * (na * ng * (nb + nf))).sum() * p
            fl += ((m1 | m2 | m3 | m4).any(0) * ng[0]).sum() * p * nabf[b] * nb
            total += 2.0 * fl * weight * stride
    return total


def work(case):
    c, op = case, case["op"]
    if op == "term":
        n, m, p, q = c["nao"], c["nao2"], c["nabf"], c["nabf2"]
        return {"bytes": 8.0 * (p * n * n + p * q + q * m * m + 2 * n * m),
                "flops": 2.0 * (p * q * m * m + p * m * m * n + p * n * n * m)}
    if op == "batch":
        w = [work(dict(x, op="scf")) for x in _cells(c)]
        return {k: sum(x[k] for x in w) for k in ("bytes", "flops")}
    sys_ = _system(c)
    nao, nabf = sys_[3].astype(np.float64), sys_[4].astype(np.float64)

    def elements(which):
        k = _pairs(sys_, c["cut_" + which])[0]
        i, j = k[:, 0], k[:, 1]
        return float({"C": nabf[i] * nao[i] * nao[j], "V": nabf[i] * nabf[j],
                      "D": nao[i] * nao[j]}[which].sum())
    if op == "density":
        nb, nk = nao.sum(), c["nk"] ** 3
        nbands = min(nb, math.ceil(2.5 * len(nao)))
        out = elements("D")
        return {"bytes": 8.0 * (nk * nb * nbands * 2 + nk * nbands + out),
                "flops": 8.0 * nk * nb * nb * nbands + 4.0 * nk * out}
    if op == "sigma_k":
        nb, nk = nao.sum(), c["nk"] ** 3
        return {"bytes": 16.0 * nk * nb * nb, "flops": 4.0 * nk * nb * nb}
    size = 8.0 * (elements("C") + elements("V") + 2.0 * elements("D"))
    if op == "grad":  # the gradients have the size of C and V, and about twice the work of the build
        return {"bytes": 2.0 * size, "flops": 3.0 * _counts(c)}
    return {"bytes": size, "flops": _counts(c)}


# ------------------------------------------------------------------- the same in 64 bits, by torch

class _Dense:
    """A cell's blocks padded to the largest sizes, with key lookup by table, and its sums."""

    def __init__(self, c, sys_, b):
        self.c, self.nao, self.nabf = c, sys_[3], sys_[4]
        self.nat, self.N, self.P = len(sys_[3]), int(sys_[3].max()), int(sys_[4].max())
        self.keys = {k: torch.from_numpy(b[k].keys.astype(np.int64)).cuda() for k in "CVD"}
        self.mask = {k: self._mask(k, b[k].keys) for k in "CVD"}
        self.pad = {}
        for k in "CVD":
            x = torch.zeros(self.mask[k].shape, dtype=torch.float64, device="cuda")
            x[self.mask[k]] = b[k].data
            self.pad[k] = x
        self.mx = {k: self.pad[k].abs().flatten(1).amax(1) for k in "CVD"}
        self.start = np.searchsorted(b["C"].keys[:, 0], np.arange(self.nat + 1))
        self.hkV, self.dR = b["V"].keys, int(np.abs(b["D"].keys[:, 2:]).max())
        side = 2 * self.dR + 1
        self.dtab = torch.full((self.nat, self.nat, side, side, side), -1, device="cuda")
        k = self.keys["D"]
        self.dtab[k[:, 0], k[:, 1], k[:, 2] + self.dR, k[:, 3] + self.dR, k[:, 4] + self.dR] = \
            torch.arange(len(k), device="cuda")
        self.eri = self._eri(b) if c["eri"] >= 0.0 else None

    def _mask(self, which, keys):
        a, f = torch.from_numpy(self.nao).cuda(), torch.from_numpy(self.nabf).cuda()
        i, j = (torch.from_numpy(keys[:, t].astype(np.int64)).cuda() for t in (0, 1))
        ab = lambda n, m: torch.arange(m, device="cuda") < n[:, None]  # noqa: E731
        if which == "V":
            return ab(f[i], self.P)[:, :, None] & ab(f[j], self.P)[:, None, :]
        m = ab(a[i], self.N)[:, :, None] & ab(a[j], self.N)[:, None, :]
        return m if which == "D" else ab(f[i], self.P)[:, :, None, None] & m[:, None]

    def dfind(self, i, j, n):
        i, j = torch.broadcast_tensors(i, j)
        ok = (n.abs() <= self.dR).all(-1)
        q = n.clamp(-self.dR, self.dR) + self.dR
        return torch.where(ok, self.dtab[i, j, q[..., 0], q[..., 1], q[..., 2]], -1)

    def _eri(self, b):
        """sqrt(max(Q, 0)) of every C block: the largest diagonal ERI of its orbital pairs."""
        at = {k: {tuple(q): e for e, q in enumerate(b[k].keys.tolist())} for k in "CV"}
        C, V = self.pad["C"], self.pad["V"]
        zero = torch.zeros(self.P, self.P, dtype=torch.float64, device="cuda")
        v = lambda *k: V[at["V"][k]] if k in at["V"] else zero  # noqa: E731
        out = []
        for e, (x, y, p, q, r) in enumerate(b["C"].keys.tolist()):
            u = C[e].flatten(1)
            t = (u * (v(x, x, 0, 0, 0) @ u)).sum(0)
            other = at["C"].get((y, x, -p, -q, -r))
            if (x, y, p, q, r) != (x, x, 0, 0, 0) and other is not None:
                w = C[other].transpose(1, 2).flatten(1)
                t = t + (u * (v(x, y, p, q, r) @ w)).sum(0) + (w * (v(y, x, -p, -q, -r) @ u)).sum(0) \
                    + (w * (v(y, y, 0, 0, 0) @ w)).sum(0)
            live = self.mask["C"][e].any(0).flatten()
            out.append(t[live].max().clamp(min=0.0).sqrt())
        return torch.stack(out)

    def pairs(self, half=False):
        """Per V block (half: of two mirrors the first): the surviving masks over the active F and G,
        and the gathered blocks."""
        kc, kd, mc, md = self.keys["C"], self.pad["D"], self.mx["C"], self.mx["D"]
        for e, (a, b, n0, n1, n2) in enumerate(self.hkV.tolist()):
            if half and (a, b, n0, n1, n2) > (b, a, -n0, -n1, -n2):
                continue
            n = torch.tensor([n0, n1, n2], device="cuda")
            fe = torch.arange(self.start[a], self.start[a + 1], device="cuda")
            ge = torch.arange(self.start[b], self.start[b + 1], device="cuda")
            f, mf, g, mg = kc[fe, 1], kc[fe, 2:], kc[ge, 1], kc[ge, 2:] + n
            A, B = torch.tensor(a, device="cuda"), torch.tensor(b, device="cuda")
            dFG = self.dfind(f[:, None], g[None], mg[None] - mf[:, None])
            dFB, dAG, dAB = self.dfind(f, B, n - mf), self.dfind(A, g, mg), self.dfind(A, B, n)
            cc, mv = mc[fe][:, None] * mc[ge][None], self.mx["V"][e]
            big = lambda d: torch.where(d >= 0, mv * md[d.clamp(min=0)], -1.0)  # noqa: E731
            far = ((f != a) | (mf != 0).any(1))[:, None]
            gar = ((g != b) | (mg != n).any(1))[None]
            th = self.c["theta"]
            m = [cc * big(dFG) > th, (cc * big(dFB)[:, None] > th) & gar,
                 (cc * big(dAG)[None] > th) & far, (cc * big(dAB) > th) & far & gar]
            if self.eri is not None:
                keep = self.eri[fe][:, None] * self.eri[ge][None] > self.c["eri"]
                m = [x & keep for x in m]
            some = m[0] | m[1] | m[2] | m[3]
            fs, gs = some.any(1).nonzero()[:, 0], some.any(0).nonzero()[:, 0]
            if not len(fs):
                continue
            m = [x[fs][:, gs].double() for x in m]
            blk = lambda d: kd[d.clamp(min=0)] * (d >= 0)[..., None, None]  # noqa: E731
            yield {"e": e, "a": a, "b": b, "n": n, "m": m, "fe": fe[fs], "ge": ge[gs], "f": f[fs],
                   "g": g[gs], "mf": mf[fs], "mg": mg[gs], "V": self.pad["V"][e],
                   "CF": self.pad["C"][fe[fs]], "CG": self.pad["C"][ge[gs]],
                   "FG": blk(dFG[fs][:, gs]), "FB": blk(dFB[fs]), "AG": blk(dAG[gs]), "AB": blk(dAB)}

    def sigma(self):
        """(keys, values, E_X) of the exchange matrix of the surviving terms."""
        N, P, nat = self.N, self.P, self.nat
        R = int(np.abs(self.hkV[:, 2:]).max()) + 2 * int(self.keys["C"][:, 2:].abs().max())
        side = 2 * R + 1
        acc = torch.zeros(nat * nat * side ** 3, N, N, dtype=torch.float64, device="cuda")
        hit = torch.zeros(nat * nat * side ** 3, dtype=torch.bool, device="cuda")

        def row(i, j, n):
            return (((i * nat + j) * side + n[..., 0] + R) * side + n[..., 1] + R) * side + n[..., 2] + R

        def add(at, x, live):
            acc.index_add_(0, at[live], -w * x[live])
            hit[at[live]] = True
        # V and D are Hermitian: a pair's mirror gives the transposed terms, added at the end
        for p in self.pairs(half=True):
            w = 0.5 if p["a"] == p["b"] and not bool(p["n"].any()) else 1.0
            m1, m2, m3, m4 = p["m"]
            nF, nG = m1.shape
            CF = p["CF"].permute(1, 2, 0, 3)                                         # al a F f
            Y = (p["V"] @ p["CG"].permute(1, 2, 0, 3).reshape(P, -1)).view(P, N, nG, N)  # al b G g
            T = Y.reshape(P * N, -1) @ (p["FG"] * m1[..., None, None]).permute(1, 3, 0, 2).reshape(nG * N, -1)
            s1 = CF.permute(1, 0, 2, 3).reshape(N, -1) @ T.view(P, N, -1).permute(0, 2, 1).reshape(-1, N)
            A, B = (torch.tensor([p[k]], device="cuda") for k in "ab")
            add(row(A, B, p["n"][None]), s1[None], (m1.sum() > 0)[None])
            Q = (p["CF"].reshape(nF, P * N, N) @ p["FB"]).reshape(nF, -1)            # F al a b
            Qs = (m2.T @ Q).view(nG, P, N, N).permute(0, 2, 1, 3).reshape(nG, N, -1)  # G a (al b)
            add(row(A, p["g"], p["mg"]), Qs @ Y.permute(2, 0, 1, 3).reshape(nG, -1, N), m2.sum(0) > 0)
            T3 = torch.einsum("xbGg,Gag->Gxab", Y, p["AG"]).reshape(nG, -1)
            Ts = (m3 @ T3).view(nF, P * N, N)
            add(row(p["f"], B, p["n"] - p["mf"]), p["CF"].reshape(nF, P * N, N).transpose(1, 2) @ Ts,
                m3.sum(1) > 0)
            Pm = torch.einsum("ab,xbGg->xaGg", p["AB"], Y).reshape(P * N, -1)
            s4 = (CF.reshape(P * N, -1).T @ Pm).view(nF, N, nG, N).permute(0, 2, 1, 3).reshape(-1, N, N)
            add(row(p["f"][:, None], p["g"][None], p["mg"][None] - p["mf"][:, None]).reshape(-1), s4,
                m4.reshape(-1) > 0)
        acc = acc.view(nat, nat, side ** 3, N, N)
        hit = hit.view(nat, nat, side ** 3)
        hit = hit | hit.transpose(0, 1).flip(2)
        at = hit.nonzero()
        i, j, t = at[:, 0], at[:, 1], at[:, 2]
        val = acc[i, j, t] + acc[j, i, side ** 3 - 1 - t].transpose(1, 2)
        del acc
        n = torch.stack([t // side ** 2, t // side % side, t % side], 1) - R
        keys = torch.cat([at[:, :2], n], 1)
        d = self.dfind(keys[:, 0], keys[:, 1], keys[:, 2:])
        ex = 0.5 * (self.pad["D"][d[d >= 0]] * val[d >= 0]).sum()
        keys = keys.cpu().numpy().astype(np.int32)
        return keys, val[self._mask("D", keys)], ex

    def gradient(self):
        """(E_X, dE/dC, dE/dV) with the surviving terms held fixed."""
        N, P = self.N, self.P
        dC, dV = torch.zeros_like(self.pad["C"]), torch.zeros_like(self.pad["V"])
        for p in self.pairs():
            w14, w23 = p["m"][0] + p["m"][3], p["m"][1] + p["m"][2]
            nF, nG = w14.shape
            FG = p["FG"] * w14[..., None, None]
            Y = torch.einsum("xy,Gybg->xbGg", p["V"], p["CG"])
            Z1 = torch.einsum("Fxaf,FGfg->xaGg", p["CF"], FG)
            Z2 = (w23.T @ (p["CF"].reshape(nF, P * N, N) @ p["FB"]).reshape(nF, -1)).view(nG, P, N, N)
            Rm = torch.einsum("ab,xaGg->xbGg", p["AB"], Z1) + torch.einsum("Gag,Gxab->xbGg", p["AG"], Z2)
            dV[p["e"]] -= 0.5 * torch.einsum("Gybg,xbGg->xy", p["CG"], Rm)
            dC.index_add_(0, p["ge"], torch.einsum("xy,xbGg->Gybg", p["V"], Rm), alpha=-0.5)
            T1 = torch.einsum("xbGg,FGfg->xbFf", Y, FG)
            Ts = (w23 @ torch.einsum("xbGg,Gag->Gxab", Y, p["AG"]).reshape(nG, -1)).view(nF, P, N, N)
            dC.index_add_(0, p["fe"], torch.einsum("ab,xbFf->Fxaf", p["AB"], T1) +
                          torch.einsum("Ffb,Fxab->Fxaf", p["FB"], Ts), alpha=-0.5)
        ex = (dV * self.pad["V"]).sum()
        return ex, dC[self.mask["C"]], dV[self.mask["V"]]


def _flat(sys_, keys):
    """Row and column of the k-space matrix, and key, of every value of a packed block set."""
    nao = sys_[3].astype(np.int64)
    first = np.concatenate([[0], np.cumsum(nao)])
    i, j = keys[:, 0], keys[:, 1]
    size = nao[i] * nao[j]
    e = np.repeat(np.arange(len(keys)), size)
    t = np.arange(size.sum()) - np.repeat(np.concatenate([[0], np.cumsum(size)[:-1]]), size)
    return first[i[e]] + t // nao[j[e]], first[j[e]] + t % nao[j[e]], e


def _long(c):
    """Whether the dense sums of a cell take too long without the library (over about 15 s)."""
    sys_ = _system(c)
    n, wide, p = len(sys_[3]), float(sys_[3].max()), float(sys_[4].max())
    nf = len(_pairs(sys_, c["cut_C"])[0]) / n
    return len(_pairs(sys_, c["cut_V"])[0]) / 2 * 6.0 * p * wide * (nf * wide) ** 2 > 1.6e13 / c.get("ncells", 1)


def exact(case, seed):
    c, op = case, case["op"]
    if op == "term":
        s = prepare(c, seed)
        return torch.einsum("xik,xy,yjl,kl->ij", s["cA"], s["V"], s["cB"], s["D"])
    if op == "density":
        sys_ = _system(c)
        kf, coef, occ = _orbitals(c, sys_, seed)
        keys = _pairs(sys_, c["cut_D"])[0]
        r, q, e = (torch.from_numpy(x).cuda() for x in _flat(sys_, keys))
        out = torch.zeros(len(r), dtype=torch.float64, device="cuda")
        for k in range(len(kf)):
            z = torch.from_numpy(coef[k]).cuda()
            rho = (z * torch.from_numpy(occ[k]).cuda()) @ z.conj().T
            ph = np.exp(2j * np.pi * (keys[:, 2:] @ kf[k]))
            out += (rho[r, q] * torch.from_numpy(ph).cuda()[e]).real
        return out / len(kf)
    if op == "batch":
        got = []
        for q, cell in enumerate(_cells(c)):
            if _long(cell):
                return None
            got.append(_Dense(cell, *_inputs(cell, 100 * int(seed) + q)).sigma())
        return {"ex": np.array([float(x[2]) for x in got]), "sigma": [x[1] for x in got]}
    if _long(c):
        return None
    sys_, b = _inputs(c, seed)
    dense = _Dense(c, sys_, b)
    if op == "grad":
        ex, dC, dV = dense.gradient()
        return {"ex": ex, "dC": dC, "dV": dV}
    keys, val, ex = dense.sigma()
    if op != "sigma_k" and c["eri"] < 0.0:
        return {"ex": float(ex), "keys": keys, "sigma": val}
    kf = _kgrid(c["nk"])
    nb = int(sys_[3].sum())
    r, q, e = (torch.from_numpy(x).cuda() for x in _flat(sys_, keys))
    out = []
    for k in kf:
        ph = torch.from_numpy(np.exp(2j * np.pi * (keys[:, 2:] @ k))).cuda()[e]
        z = torch.zeros(nb * nb, dtype=torch.complex128, device="cuda")
        out.append(z.index_add_(0, r * nb + q, val * ph).view(nb, nb))
    return torch.stack(out) if op == "sigma_k" else {"ex": float(ex), "sigma_k": torch.stack(out)}
