"""Systematic errors of the split path: rounding that is the same at every point does not average out in sums over points,
so means over many points are held to a small part of the rounding of one value."""
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
