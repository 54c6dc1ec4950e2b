"""Systematic errors: rounding that is the same at every point, or at every point of a spline segment, does not average out
in sums over points, so means over many points are held to a small part of the rounding of one value."""
import math

import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_1912_06636_gb300 import nao, synth

pytestmark = pytest.mark.gpu


def cuda(a):
    return torch.from_numpy(np.ascontiguousarray(a)).cuda()


def test_gradient_of_p_functions():
    """At x = 0 the x derivative of the p_x function is g(r) times a constant of the harmonics. Against FP64 its mean
    relative error is that constant's: one float-float, 2^-49, and a few zero-mean roundings of 2^-48 over 2000 points."""
    rng = np.random.Generator(np.random.PCG64(5))
    sp = synth.Species(ls=[1], alphas=[0.6], Z=6.0)
    s = synth.make_system([[0.0, 0.0, 0.0]], [0], [sp], n_rad=1, n_theta=1, n_phi=1)
    r, t = rng.uniform(0.3, 3.0, 2000), rng.uniform(0.0, 2.0 * np.pi, 2000)
    s.pt_xyz = np.ascontiguousarray(np.stack([0.0 * r, r * np.cos(t), r * np.sin(t)], axis=1))
    s.pt_w = np.full(2000, 0.01)
    rel = []
    with nao.Grid(s, device=0, max_batch_points=200) as g:
        for b in range(len(g.batches()[0]) - 1):
            a, x = (g.evaluate_batch(b, prec, True)[1][0, 2].cpu().numpy() for prec in ("split", "fp64"))
            rel.append(a / x - 1.0)
    assert abs(np.mean(np.concatenate(rel))) <= 2.0 ** -49 + 4 * 2.0 ** -48 / np.sqrt(2000.0)


@pytest.mark.parametrize("opts", [dict(split_slices=12), dict(split_digits=1, split_slices=14)])
def test_density_of_the_hessian(opts):
    """N_e of the split Hessian's density against the FP64 one, from the same evaluation: the values of phi that it
    multiplies are rounded to nearest, so that over 2000 points their 2^-48 average out."""
    s = synth.config_water(n_rad=20, n_theta=6, n_phi=7)
    P = cuda(synth.density_matrix(s, 4))
    with nao.Grid(s, device=0, max_batch_points=100, **opts) as g:
        ne = [float(g.density_hessian(P, prec=prec)[3].item()) for prec in ("split", "fp64")]
        g.sync()
    assert abs(ne[0] / ne[1] - 1.0) <= 1e-15


def test_radial_coordinate():
    """A steep s function in FP64 against its spline in extended precision. Its relative error over d ln phi / d ln r is
    that of ln r: sqrt(r^2) by a reciprocal root (1.5 ulp), 1 / r_k (1.5 ulp) and their product less one (half an ulp), at
    most 3.5 ulp of 1.1e-16 in all and 2e-16 in the root mean square; knots from k Delta rounded to FP64 (an ulp of 1.8e-15
    at these radii) add 5e-16."""
    ld = np.longdouble
    if np.finfo(ld).nmant < 60:
        pytest.skip("no extended precision on this host")
    rng = np.random.Generator(np.random.PCG64(6))
    sp = synth.Species(ls=[0], alphas=[3.0], Z=6.0)
    s = synth.make_system([[0.0, 0.0, 0.0]], [0], [sp], n_rad=1, n_theta=1, n_phi=1)
    d = rng.normal(size=(4000, 3))
    s.pt_xyz = np.ascontiguousarray(d * (rng.uniform(1.5, 3.0, 4000) / np.linalg.norm(d, axis=1))[:, None])
    s.pt_w = np.full(4000, 0.01)
    coef = nao.nao_radial_spline(s.fn_table[0]).astype(ld)
    delta = ld(math.log(s.r_last / s.r0) / (s.n_rgrid - 1))
    shift = []
    with nao.Grid(s, device=0, max_batch_points=200) as g:
        off, perm = g.batches()[:2]
        for b in range(len(off) - 1):
            phi = g.evaluate_batch(b, "fp64", True)[0][0].cpu().numpy()
            x = s.pt_xyz[perm[off[b]:off[b + 1]]].astype(ld)
            sc = np.log(np.sqrt((x * x).sum(axis=1)) / ld(s.r0)) / delta
            k = np.floor(sc).astype(int)
            t, c = sc - k, coef[k].T
            R = ((c[3] * t + c[2]) * t + c[1]) * t + c[0]
            slope = ((3 * c[3] * t + 2 * c[2]) * t + c[1]) / (R * delta)
            shift.append((phi / (R / np.sqrt(4 * np.arccos(ld(-1)))) - 1) / slope)
    shift = np.concatenate(shift).astype(float)
    assert np.sqrt(np.mean(shift * shift)) <= 3e-16


@pytest.mark.parametrize("opts", [dict(split_slices=12), dict(split_digits=1, split_slices=15)])
def test_density_sums(opts):
    """n = sum_j T_j phi_j of the split path from its own phi, with T = P phi: T, the product and its addition are
    rounded to a few 2^-49 of a term, independently, so that the error is at most 2^-48 of the root of the sum of the
    squared terms in the root mean square (one atom with 20 functions; points outside the sphere evaluated in FP64)."""
    ld = np.longdouble
    if np.finfo(ld).nmant < 60:
        pytest.skip("no extended precision on this host")
    rng = np.random.Generator(np.random.PCG64(7))
    sp = synth.Species(ls=[0, 0, 1, 1, 2, 3], alphas=[0.4, 1.5, 0.6, 1.1, 0.8, 0.9], Z=6.0)
    s = synth.make_system([[0.1, -0.2, 0.3]], [0], [sp], n_rad=1, n_theta=1, n_phi=1)
    assert s.n_basis == 20
    d = rng.normal(size=(2000, 3))
    s.pt_xyz = np.ascontiguousarray(s.atom_xyz[0] + d * (rng.uniform(0.15, 4.0, 2000) / np.linalg.norm(d, axis=1))[:, None])
    s.pt_w = np.full(2000, 0.01)
    P = synth.density_matrix(s, 5)
    err = []
    with nao.Grid(s, device=0, max_batch_points=200, **opts) as g:
        n = g.update_density(cuda(P), prec="split")[0].cpu().numpy()
        g.sync()
        off, perm, rel_off, rel = g.batches()
        for b in range(len(off) - 1):
            phi = g.evaluate_batch(b, "split", False)[0].cpu().numpy().astype(ld)
            i = rel[rel_off[b]:rel_off[b + 1]]
            t = (P[np.ix_(i, i)].astype(ld) @ phi) * phi
            err.append((n[perm[off[b]:off[b + 1]]] - t.sum(axis=0)) / np.sqrt((t * t).sum(axis=0)))
    assert np.sqrt(np.mean(np.concatenate(err).astype(float) ** 2)) <= 2.0 ** -48
