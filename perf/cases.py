"""Performance cases of the real-space integration library: what they stand for, their inputs, one
pass of each through the public entry points, the work a pass cannot do without, and the results
in plain 64-bit torch.

A case is a dict of plain values:
  kind    what one pass is: "scf" (H, then n and N_e: one self-consistency iteration), "many" (the
          same for a grouped handle), "grad" (n, grad n, N_e), "hess" (n, grad n, the six second
          derivatives, N_e), "pulay" (the Pulay matrix elements and the forces), "bloch" (h^uc of a
          periodic cell and its Bloch sums)
  system  the geometry: "water", "diamond" (cells^3 conventional cells), "slab" (layers of n x n),
          "molecule" (atoms, geometry), "set" (molecules of lo .. hi atoms, geometry), "crystal"
          (periodic silicon, grid^3 points, k^3 k points)
  n_rad, n_theta, n_phi   integration points per atom; batch: points per batch
  prec, slices, digits, graph, scratch_mb   precision and handle options (0: the library's default)
"""
from __future__ import annotations

import functools
import math

import numpy as np
import torch

from paper_1912_06636_gb300 import nao, synth

H_TERMS = nao.NAO_TERM_POTENTIAL | nao.NAO_TERM_KINETIC


def listed():
    tight_si = dict(n_rad=60, n_theta=17, n_phi=18)    # the diamond cluster's own grid
    tight_slab = dict(n_rad=80, n_theta=14, n_phi=31)  # the slab's own grid
    serve = dict(n_rad=30, n_theta=8, n_phi=9)         # the serving stream's grid
    split12 = dict(prec="split", slices=0, digits=0)   # the library's default: 12 bf16 slices
    e4m3 = dict(prec="split", slices=14, digits=1)     # the headline setting: 14 e4m3 slices
    plain = dict(graph=0, scratch_mb=0)
    return [
        # the smallest molecule with the default options: launches and latency
        dict(name="water", kind="scf", system="water", n_rad=40, n_theta=10, n_phi=11, batch=200, **split12, **plain),
        # a request of the serving loop: its options, replayed graphs, an ordinary molecule
        dict(name="request", kind="scf", system="molecule", atoms=21, geometry=4007, **serve, batch=200, **e4m3,
             graph=1, scratch_mb=256),
        # the 64-atom cluster on its own grid, default options
        dict(name="cluster", kind="scf", system="diamond", cells=2, **tight_si, batch=300, **split12, **plain),
        # five layers of the two-species slab on its own grid, headline setting: the largest
        dict(name="slab", kind="scf", system="slab", layers=5, n=5, **tight_slab, batch=200, **e4m3, **plain),
        # molecules of very different sizes and batch sizes in one grouped handle
        dict(name="set", kind="many", system="set", molecules=12, lo=3, hi=24, geometry=3000, **serve, batch=0, **e4m3,
             **plain),
        # the binding's default precision, on one conventional cell's cluster
        dict(name="fp64", kind="scf", system="diamond", cells=1, **tight_si, batch=300, prec="fp64", slices=0, digits=0,
             **plain),
        # single precision, where 1e-6 is enough
        dict(name="fp32", kind="scf", system="diamond", cells=2, **tight_si, batch=300, prec="fp32", slices=0, digits=0,
             **plain),
        # n and grad n, as GGA functionals need them, default options, slab basis
        dict(name="gradient", kind="grad", system="slab", layers=3, n=3, **tight_slab, batch=200, **split12, **plain),
        # n, grad n and the Hessian, as forces and stresses need them
        dict(name="hessian", kind="hess", system="molecule", atoms=13, geometry=4011, n_rad=45, n_theta=10, n_phi=13,
             batch=200, **e4m3, **plain),
        # the local Pulay terms of a force step (the FP64 path; there is no split one)
        dict(name="pulay", kind="pulay", system="molecule", atoms=9, geometry=4003, **serve, batch=200, prec="fp64",
             slices=0, digits=0, **plain),
        # periodic silicon: h^uc over the image functions and h(k) on a Monkhorst-Pack mesh
        dict(name="crystal", kind="bloch", system="crystal", grid=48, k=4, batch=300, prec="split", slices=11, digits=0,
             **plain),
    ]


def _log_int(rng, lo, hi):
    return min(hi, int(math.exp(rng.uniform(math.log(lo), math.log(hi + 1)))))


def draw(rng):
    kind = rng.choice(("scf", "scf", "scf", "scf", "many", "grad", "hess", "pulay", "bloch"))
    c = dict(kind=kind, graph=rng.choice((0, 0, 1)), scratch_mb=rng.choice((0, 0, 256)))
    prec = rng.choice(("split", "split", "split", "fp64", "fp32")) if kind != "pulay" else rng.choice(("fp64", "fp32"))
    digits = rng.choice((0, 1))
    c.update(prec=prec, digits=digits, slices=rng.choice((0, 11, 12)) if digits == 0 else rng.choice((13, 14, 15)))
    if kind == "bloch":
        c.update(system="crystal", grid=_log_int(rng, 18, 44), k=rng.randint(1, 4), batch=_log_int(rng, 60, 400))
        if prec == "fp64":
            c["grid"] = min(c["grid"], 24)
        if c["grid"] % 4 == 2:  # a grid point would sit on the nuclei at 1/4 and 3/4 of the cell
            c["grid"] += 1
        return c
    c.update(n_rad=_log_int(rng, 14, 60), n_theta=rng.randint(5, 14), n_phi=rng.randint(6, 19),
             batch=_log_int(rng, 40, 400))
    if kind == "many":
        c.update(system="set", molecules=_log_int(rng, 2, 12), lo=3, hi=rng.randint(6, 16), geometry=3000 + rng.randrange(999),
                 batch=0)
        c["n_rad"] = min(c["n_rad"], 24)
    elif kind in ("scf", "grad") and rng.random() < 0.4:
        if rng.random() < 0.5:
            c.update(system="slab", layers=rng.randint(1, 4), n=rng.randint(2, 3))
        else:
            c.update(system="diamond", cells=1)
    else:
        c.update(system="molecule", atoms=_log_int(rng, 2, 40), geometry=4000 + rng.randrange(999))
    if prec == "fp64" or kind in ("hess", "pulay"):  # keeps the slow paths below the largest listed case
        c["n_rad"] = min(c["n_rad"], 24)
        if "atoms" in c:
            c["atoms"] = min(c["atoms"], 16)
    return c


# ---- inputs ---------------------------------------------------------------------------------
_SYSTEM_KEYS = ("system", "cells", "layers", "n", "atoms", "geometry", "molecules", "lo", "hi", "grid", "n_rad",
                "n_theta", "n_phi")


@functools.lru_cache(maxsize=24)
def _systems(key):
    """[(system, its potential)], the batch sizes of a set, and the images of a crystal, from the
    case's geometry alone (a user's program reads these once per geometry)."""
    c = dict(key)
    if c["system"] == "crystal":
        cell = synth.diamond_cluster(10.26, 1) / 10.26
        unit = synth.periodic_cell(10.26 * np.eye(3), cell, [0] * len(cell), [synth.silicon_species(1)], n_grid=c["grid"])
        lattice = unit.meta["lattice"]
        xyz, atom, shift = nao.nao_periodic_images(unit.atom_xyz, lattice, float(np.max(unit.fn_cutoff)))
        s = synth.image_system(unit, xyz, atom)
        fmap, fimg = nao.nao_periodic_basis_map(unit, atom)
        return [(s, synth.periodic_potential(unit))], None, (lattice, shift, fmap, fimg, unit.n_basis)
    grid = dict(n_rad=c["n_rad"], n_theta=c["n_theta"], n_phi=c["n_phi"])
    batches = None
    if c["system"] == "water":
        out = [synth.config_water(**grid)]
    elif c["system"] == "diamond":
        out = [synth.config_diamond64(cells=c["cells"], **grid)]
    elif c["system"] == "slab":
        out = [synth.config_slab375(layers=c["layers"], n=c["n"], **grid)]
    elif c["system"] == "molecule":
        out = [synth.random_molecule(c["atoms"], c["geometry"], **grid)]
    else:
        out, batches = synth.molecule_set(c["molecules"], seed=c["geometry"], n_min=c["lo"], n_max=c["hi"], **grid)
    return [(s, s.potential(on_device=True)) for s in out], batches, None


def _inputs(case, seed):
    """(systems, v per system, P per system (two of them for the Pulay terms), batch sizes, crystal):
    the potential moves by 1 % per point from one iteration to the next, P is a new density matrix."""
    systems, batches, crystal = _systems(tuple(sorted((k, case[k]) for k in _SYSTEM_KEYS if k in case)))
    gen = torch.Generator(device="cuda").manual_seed(int(seed))
    vs, ps = [], []
    for s, v0 in systems:
        v = torch.as_tensor(v0, dtype=torch.float64, device="cuda")
        vs.append(v * (1.0 + 0.01 * (2.0 * torch.rand(v.shape, generator=gen, dtype=torch.float64, device="cuda") - 1.0)))
        for _ in range(2 if case["kind"] == "pulay" else 0 if case["kind"] == "bloch" else 1):
            x = torch.randn((s.n_basis, 16), generator=gen, dtype=torch.float64, device="cuda")
            p = x @ x.T / 16.0
            ps.append(0.5 * (p + p.T))
    return [s for s, _ in systems], vs, ps, batches, crystal


def _grid(case, systems, batches):
    opts = dict(split_digits=case["digits"], capture_graph=case["graph"])
    if case["slices"]:
        opts["split_slices"] = case["slices"]
    if case["scratch_mb"]:
        opts["scratch_bytes"] = case["scratch_mb"] << 20
    if case["kind"] == "many":
        return nao.Grid(systems, batch_points=batches, **opts)
    return nao.Grid(systems[0], max_batch_points=case["batch"], **opts)


def _empty(*shape):
    return torch.empty(shape, dtype=torch.float64, device="cuda")


def prepare(case, seed):
    systems, vs, ps, batches, crystal = _inputs(case, seed)
    st = dict(kind=case["kind"], prec=case["prec"], g=_grid(case, systems, batches), v=vs, p=ps)
    nb, n_pts = [s.n_basis for s in systems], [s.n_points for s in systems]
    if case["kind"] in ("scf", "many", "bloch"):
        st["H"] = [_empty(b, b) for b in nb]
    if case["kind"] in ("scf", "many", "grad", "hess"):
        st["n"] = [_empty(p) for p in n_pts]
        st["ne"] = [_empty(1) for _ in nb]
    if case["kind"] in ("grad", "hess"):
        st["grad"] = _empty(3, n_pts[0])
    if case["kind"] == "hess":
        st["hess"] = _empty(6, n_pts[0])
    if case["kind"] == "pulay":
        st["M"], st["S"], st["F"] = _empty(3, nb[0], nb[0]), _empty(3, nb[0], nb[0]), _empty(systems[0].n_atoms, 3)
    if case["kind"] == "bloch":
        lattice, shift, fmap, fimg, n_cell = crystal
        st.update(lattice=lattice, nb=n_cell, k=torch.as_tensor(_k_points(lattice, case["k"]), device="cuda"),
                  fmap=torch.as_tensor(fmap, device="cuda"), fimg=torch.as_tensor(fimg, device="cuda"),
                  shift=torch.as_tensor(shift, device="cuda"), hk=_empty(case["k"] ** 3, n_cell, n_cell, 2))
    return st


def _k_points(lattice, k):
    f = (np.arange(k) + 0.5) / k - 0.5
    fr = np.stack(np.meshgrid(f, f, f, indexing="ij"), axis=-1).reshape(-1, 3)
    return fr @ (2.0 * math.pi * np.linalg.inv(lattice).T)


def run(st):
    g, prec, kind = st["g"], st["prec"], st["kind"]
    if kind == "scf":
        H = g.integrate_h(st["v"][0], H_TERMS, prec, st["H"][0])
        n, ne = g.update_density(st["p"][0], prec, st["n"][0], st["ne"][0])
        return {"H": H, "n": n, "ne": ne}
    if kind == "many":
        H = g.integrate_h_many(st["v"], H_TERMS, prec, st["H"])
        n, ne = g.update_density_many(st["p"], prec, st["n"], st["ne"])
        return {"H": H, "n": n, "ne": ne}
    if kind == "grad":
        n, gn, ne = g.density_gradient(st["p"][0], prec, st["n"][0], st["grad"], st["ne"][0])
        return {"n": n, "grad": gn, "ne": ne}
    if kind == "hess":
        n, gn, h, ne = g.density_hessian(st["p"][0], prec, st["n"][0], st["grad"], st["hess"], st["ne"][0])
        return {"n": n, "grad": gn, "hess": h, "ne": ne}
    if kind == "pulay":
        M, S = g.pulay_matrices(st["v"][0], prec, st["M"], st["S"])
        return {"M": M, "S": S, "F": g.pulay_forces(st["p"][0], st["p"][1], M, S, st["F"])}
    H = g.integrate_h(st["v"][0], H_TERMS, prec, st["H"][0])
    return {"H": H, "hk": nao.nao_bloch_sum(H, st["fmap"], st["fimg"], st["shift"], st["lattice"], st["k"], st["nb"],
                                            out=st["hk"])}


def work(case):
    """Operations of the batch products over the reduced bases (the handle's own counts); bytes of
    the points, weights, potential, radial tables and matrices that go in and of what comes out."""
    systems, _, _, batches, _ = _inputs(case, 0)
    with _grid(case, systems, batches) as g:
        fh, fn = float(g.info.flops_h), float(g.info.flops_n)  # 4 P N (N + 1) and 2 P N^2 + 2 P N, summed
        pts, nb2 = float(g.n_points), float(sum(s.n_basis ** 2 for s in systems))
    table = float(sum(s.fn_table.size for s in systems)) * 8.0
    base = 32.0 * pts + table
    kind = case["kind"]
    if kind in ("scf", "many"):
        return {"bytes": base + 16.0 * pts + 16.0 * nb2, "flops": fh + fn}
    if kind == "grad":
        return {"bytes": base + 32.0 * pts + 8.0 * nb2, "flops": 2.0 * fn}
    if kind == "hess":
        return {"bytes": base + 80.0 * pts + 8.0 * nb2, "flops": 4.0 * fn}
    if kind == "pulay":
        return {"bytes": base + 8.0 * pts + 8.0 * nb2 * 8.0, "flops": 3.0 * fh + 12.0 * nb2}
    n_cell, nk = float(8 * 25), float(case["k"] ** 3)
    return {"bytes": base + 8.0 * pts + 8.0 * nb2 + 16.0 * nk * n_cell ** 2, "flops": fh + 8.0 * nk * nb2}


# ---- the same results in plain 64-bit torch ---------------------------------------------------
# phi = g(r) S(x, y, z), g = R / r^l, R the natural cubic spline in s = ln(r / r0) / Delta through
# the table, S the real solid harmonics as polynomials in x, y, z; derivatives by the product rule.
def _pmul(a, b):
    out = {}
    for (i, j, k), u in a.items():
        for (p, q, r), w in b.items():
            e = (i + p, j + q, k + r)
            out[e] = out.get(e, 0.0) + u * w
    return out


def _padd(a, b, fa=1.0, fb=1.0):
    out = {e: fa * u for e, u in a.items()}
    for e, u in b.items():
        out[e] = out.get(e, 0.0) + fb * u
    return {e: u for e, u in out.items() if u != 0.0}


def _pdiff(a, axis):
    out = {}
    for e, u in a.items():
        if e[axis]:
            d = list(e)
            d[axis] -= 1
            out[tuple(d)] = out.get(tuple(d), 0.0) + u * e[axis]
    return out


@functools.lru_cache(maxsize=None)
def _harmonics(l):
    """S_lm, m = -l .. l, as {(i, j, k): coefficient of x^i y^j z^k}."""
    z, r2 = {(0, 0, 1): 1.0}, {(2, 0, 0): 1.0, (0, 2, 0): 1.0, (0, 0, 2): 1.0}
    ab = [({(0, 0, 0): 1.0}, {})]  # real and imaginary part of (x + i y)^m
    for _ in range(l):
        a, b = ab[-1]
        x, y = {(1, 0, 0): 1.0}, {(0, 1, 0): 1.0}
        ab.append((_padd(_pmul(x, a), _pmul(y, b), 1.0, -1.0), _padd(_pmul(x, b), _pmul(y, a))))
    out = [None] * (2 * l + 1)
    for m in range(l + 1):
        df = 1.0
        for q in range(1, 2 * m, 2):
            df *= q
        pi = [{(0, 0, 0): df}]  # r^(q - m) P_q^m / sin^m, q = m, m + 1, ..
        for q in range(m + 1, l + 1):
            t = _pmul(z, pi[-1])
            t = {e: u * (2 * q - 1) / (q - m) for e, u in t.items()}
            if q - m >= 2:
                t = _padd(t, _pmul(r2, pi[-2]), 1.0, -(q + m - 1) / (q - m))
            pi.append(t)
        k = math.sqrt((2 * l + 1) / (4 * math.pi) * math.factorial(l - m) / math.factorial(l + m) * (2.0 if m else 1.0))
        for sign in ((1, -1) if m else (1,)):
            out[l + sign * m] = {e: k * u for e, u in _pmul(pi[-1], ab[m][0 if sign > 0 else 1]).items()}
    return out


def _poly(p, x):
    """A polynomial at x = [powers of x, of y, of z]."""
    out = torch.zeros_like(x[0][0])
    for (i, j, k), u in p.items():
        out = out + u * (x[0][i] * x[1][j] * x[2][k])
    return out


def _spline(table):
    """[n_fn, n - 1, 4] coefficients of the natural cubic splines through the rows of the table."""
    n = table.shape[1]
    a = 4.0 * np.eye(n - 2) + np.eye(n - 2, k=1) + np.eye(n - 2, k=-1)
    m = np.zeros_like(table)  # second derivatives
    m[:, 1:-1] = np.linalg.solve(a, 6.0 * (table[:, 2:] - 2.0 * table[:, 1:-1] + table[:, :-2]).T).T
    y0, y1, m0, m1 = table[:, :-1], table[:, 1:], m[:, :-1], m[:, 1:]
    return np.stack([y0, y1 - y0 - (2.0 * m0 + m1) / 6.0, m0 / 2.0, (m1 - m0) / 6.0], axis=-1)


class _Exact:
    """The basis of one system in blocks of nearby points."""

    def __init__(self, s):
        self.s = s
        self.dev = "cuda" if torch.cuda.is_available() else "cpu"
        t = lambda a: torch.as_tensor(np.ascontiguousarray(a), dtype=torch.float64, device=self.dev)  # noqa: E731
        self.xyz, self.pts, self.w = t(s.atom_xyz), t(s.pt_xyz), t(s.pt_w)
        self.coef = t(_spline(np.asarray(s.fn_table)))
        self.delta = math.log(s.r_last / s.r0) / (s.n_rgrid - 1)
        self.spec = np.asarray(s.atom_species)
        off = s.species_fn_offset
        self.fns = [range(int(off[k]), int(off[k + 1])) for k in range(len(off) - 1)]
        size = [sum(2 * int(s.fn_l[f]) + 1 for f in fs) for fs in self.fns]
        self.first = np.concatenate([[0], np.cumsum([size[k] for k in self.spec])])
        self.size = size

    def blocks(self, edge=4.0, most=6000):
        """(points, relevant atoms per species) of cubes of space; points that no function reaches are left out."""
        rc = float(np.max(self.s.fn_cutoff))
        near = torch.cat([(torch.cdist(p, self.xyz) < rc).any(dim=1) for p in self.pts.split(200000)])
        idx = near.nonzero()[:, 0]
        lo = self.xyz.min(dim=0).values - rc
        cell = ((self.pts[idx] - lo) / edge).floor().to(torch.int64)
        key = (cell[:, 0] * 4096 + cell[:, 1]) * 4096 + cell[:, 2]
        order = torch.argsort(key, stable=True)
        idx, key = idx[order], key[order]
        _, count = torch.unique_consecutive(key, return_counts=True)
        at = 0
        for c in count.tolist():
            for b in range(at, at + c, most):
                q = idx[b:min(b + most, at + c)]
                x = self.pts[q]
                gap = torch.clamp(torch.maximum(x.min(dim=0).values - self.xyz, self.xyz - x.max(dim=0).values), min=0.0)
                hit = ((gap * gap).sum(dim=1) < rc * rc).cpu().numpy()
                yield q, [np.flatnonzero(hit & (self.spec == k)) for k in range(len(self.fns))]
            at += c

    def basis(self, q, atoms, order):
        """Global function indices [N] and values [1, 4 or 10][N, points] (phi; d_x, d_y, d_z; xx, xy, xz, yy, yz, zz)."""
        idx, rows = [], []
        for sp, at in enumerate(atoms):
            if not len(at):
                continue
            d = self.pts[q][None, :, :] - self.xyz[torch.as_tensor(at, device=self.dev)][:, None, :]
            x = [d[..., c] for c in range(3)]
            r = torch.sqrt((d * d).sum(dim=-1))
            rr = torch.clamp(r, min=self.s.r0)
            sc = torch.log(rr / self.s.r0) / self.delta
            k = torch.clamp(sc.floor().to(torch.int64), 0, self.s.n_rgrid - 2)
            t = sc - k
            d1, d2 = 1.0 / (self.delta * rr), -1.0 / (self.delta * rr * rr)
            ls = [int(self.s.fn_l[f]) for f in self.fns[sp]]
            pw = [[torch.ones_like(r)] for _ in range(3)]
            for c in range(3):
                for _ in range(max(ls)):
                    pw[c].append(pw[c][-1] * x[c])
            harm = {}
            pos = 0
            for f, l in zip(self.fns[sp], ls):
                if l not in harm:
                    harm[l] = []
                    for p in _harmonics(l):
                        d_ = [_pdiff(p, a) for a in range(3)] if order >= 1 else []
                        dd = [_pdiff(d_[a], b) for a in range(3) for b in range(a, 3)] if order >= 2 else []
                        harm[l].append([_poly(u, pw) for u in [p] + d_ + dd])
                cf = self.coef[f][k]
                c0, c1, c2, c3 = (cf[..., i] for i in range(4))
                inside = (r < float(self.s.fn_cutoff[f])).to(torch.float64)
                R = (((c3 * t + c2) * t + c1) * t + c0) * inside
                g = R / r ** l
                if order >= 1:
                    Rs = ((3.0 * c3 * t + 2.0 * c2) * t + c1) * inside
                    R1 = Rs * d1
                    g1 = (R1 - l * R / r) / r ** l
                if order >= 2:
                    R2 = (6.0 * c3 * t + 2.0 * c2) * inside * d1 * d1 + Rs * d2
                    g2 = (R2 - 2.0 * l * R1 / r + l * (l + 1) * R / (r * r)) / r ** l
                for m, h in enumerate(harm[l]):
                    v = [g * h[0]]
                    if order >= 1:
                        v += [g1 / r * x[a] * h[0] + g * h[1 + a] for a in range(3)]
                    if order >= 2:
                        u = 4
                        for a in range(3):
                            for b in range(a, 3):
                                t2 = (g2 - g1 / r) / (r * r) * x[a] * x[b] * h[0]
                                t2 = t2 + g1 / r * ((h[0] if a == b else 0.0) + x[b] * h[1 + a] + x[a] * h[1 + b])
                                v.append(t2 + g * h[u])
                                u += 1
                    rows.append(torch.stack(v))
                    idx.append(self.first[at] + pos + m)
                pos += 2 * l + 1
        if not rows:
            return None, None
        i = torch.as_tensor(np.concatenate(idx), device=self.dev)
        return i, torch.cat(rows, dim=1)


def _exact_one(s, v, ps, kind):
    ex = _Exact(s)
    order = 2 if kind in ("hess", "pulay") else 1
    nb, n_pts = s.n_basis, s.n_points
    zeros = lambda *sh: torch.zeros(sh, dtype=torch.float64, device=ex.dev)  # noqa: E731
    H, n, gn, hs, M, S = zeros(nb, nb), zeros(n_pts), zeros(3, n_pts), zeros(6, n_pts), None, None
    if kind == "pulay":
        M, S = zeros(3, nb, nb), zeros(3, nb, nb)
    for q, atoms in ex.blocks():
        i, E = ex.basis(q, atoms, order)
        if i is None:
            continue
        w = ex.w[q]
        if kind in ("scf", "many", "bloch"):
            h = (E[0] * (w * v[q])) @ E[0].T
            for c in range(3):
                h += (E[1 + c] * (0.5 * w)) @ E[1 + c].T
            H[i[:, None], i] += h
        if kind in ("scf", "many", "grad", "hess"):
            T = ps[0][i][:, i] @ E[0]
            n[q] = (T * E[0]).sum(dim=0)
            if kind in ("grad", "hess"):
                for c in range(3):
                    gn[c, q] = 2.0 * (T * E[1 + c]).sum(dim=0)
            if kind == "hess":
                Tc = [ps[0][i][:, i] @ E[1 + c] for c in range(3)]
                pairs = [(a, b) for a in range(3) for b in range(a, 3)]
                for k, (a, b) in enumerate(pairs):
                    hs[k, q] = 2.0 * ((T * E[4 + k]).sum(dim=0) + (Tc[a] * E[1 + b]).sum(dim=0))
        if kind == "pulay":
            hphi = -0.5 * (E[4] + E[7] + E[9]) + v[q] * E[0]
            for c in range(3):
                M[c][i[:, None], i] += (w * E[1 + c]) @ hphi.T
                S[c][i[:, None], i] += (w * E[1 + c]) @ E[0].T
    ne = (ex.w * n).sum().reshape(1)
    if kind == "grad":
        return {"n": n, "grad": gn, "ne": ne}
    if kind == "hess":
        return {"n": n, "grad": gn, "hess": hs, "ne": ne}
    if kind == "pulay":
        f = 2.0 * (ps[0] * M - ps[1] * S).sum(dim=2)  # [3, nb]
        at = torch.as_tensor(np.repeat(np.arange(s.n_atoms), np.diff(ex.first)), device=ex.dev)
        return {"M": M, "S": S, "F": zeros(s.n_atoms, 3).index_add_(0, at, f.T.contiguous())}
    return {"H": H, "n": n, "ne": ne}


def exact(case, seed):
    systems, vs, ps, _, crystal = _inputs(case, seed)
    kind = case["kind"]
    if kind == "many":
        each = [_exact_one(s, v, [p], "many") for s, v, p in zip(systems, vs, ps)]
        return {k: [e[k] for e in each] for k in ("H", "n", "ne")}
    got = _exact_one(systems[0], vs[0], ps, kind)
    if kind != "bloch":
        return got
    lattice, shift, fmap, fimg, n_cell = crystal
    H = got["H"]
    T = torch.as_tensor((shift.astype(np.float64) @ lattice)[fimg], device=H.device)
    to = torch.as_tensor(fmap.astype(np.int64), device=H.device)
    hk = []
    for k in torch.as_tensor(_k_points(lattice, case["k"]), device=H.device):
        ph = torch.polar(torch.ones_like(T[:, 0]), T @ k)
        h = H * (ph.conj()[:, None] * ph[None, :])
        rows = torch.zeros((n_cell, h.shape[1]), dtype=h.dtype, device=H.device).index_add_(0, to, h)
        hk.append(torch.zeros((n_cell, n_cell), dtype=h.dtype, device=H.device).index_add_(1, to, rows))
    return {"H": H, "hk": torch.stack(hk)}
