"""Points closer to a nucleus than the first knot r0 of the radial grid, where the radial functions and both of
their derivatives are those at r0: density, its gradient and Hessian and the Pulay matrices against the oracle, at
the bars of the other parity tests (FP64 1e-12, FP32 1e-6, split 1e-10 of the magnitude sums)."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

import oracle
from paper_1912_06636_gb300 import nao, synth
from tests._metrics import rel_err

pytestmark = pytest.mark.gpu

TOL = {"fp64": 1e-12, "fp32": 1e-6, "split": 1e-10}


def cuda(a):
    return torch.from_numpy(np.ascontiguousarray(a)).cuda()


def inner_points(ls, r0):
    """One atom with the functions ls, points at 0.02, 0.3 and 0.9 r0 and four times as many farther out."""
    rng = np.random.Generator(np.random.PCG64(11))
    sp = synth.Species(ls=list(ls), alphas=[0.7 + 0.4 * k for k in range(len(ls))], Z=6.0)
    s = synth.make_system([[0.0, 0.0, 0.0]], [0], [sp], n_rad=1, n_theta=1, n_phi=1, r0=r0)
    d = rng.normal(size=(150, 3))
    d /= np.linalg.norm(d, axis=1)[:, None]
    r = np.concatenate([np.repeat([0.02, 0.3, 0.9], 10) * r0, rng.uniform(0.2, 3.0, 120)])
    s.pt_xyz = np.ascontiguousarray(d * r[:, None])
    s.pt_w = rng.uniform(0.001, 0.01, 150)
    return s


@pytest.mark.parametrize("r0", [1e-4, 1e-2])
@pytest.mark.parametrize("ls", [[0], [1], [2], [3], [0, 1, 2, 3, 0]])
def test_points_inside_the_first_knot(ls, r0):
    s = inner_points(ls, r0)
    o = oracle.Oracle(s)
    v, P = s.potential(), synth.density_matrix(s, 3)
    n, D, _ = o.density(s.pt_xyz, P, s.pt_w)
    gref, Dg = o.density_gradient(s.pt_xyz, P)
    href, Dh = o.density_hessian(s.pt_xyz, P)
    M, S, AM, AS = o.pulay_matrices(s.pt_xyz, s.pt_w, v)
    with nao.Grid(s, device=0, max_batch_points=40) as g:
        for prec, tol in TOL.items():
            x, gr, h, _ = (t.cpu().numpy() for t in g.density_hessian(cuda(P), prec=prec))
            g.sync()
            assert rel_err(x, n, D) <= tol, prec
            for c in range(3):
                assert rel_err(gr[c], gref[:, c], Dg[:, c]) <= tol, (prec, c)
            for k in range(6):
                assert rel_err(h[k], href[:, k], Dh[:, k]) <= tol, (prec, k)
            if prec != "split":  # at the matrices' scale, as the other Pulay tests
                m, x = (t.cpu().numpy() for t in g.pulay_matrices(cuda(v), prec=prec))
                for c in range(3):
                    assert np.max(np.abs(m[c] - M[c])) <= tol * AM[c].max(), (prec, c)
                    assert np.max(np.abs(x[c] - S[c])) <= tol * AS[c].max(), (prec, c)
