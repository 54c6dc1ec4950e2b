"""The launches that large systems and small scratch sizes take, at sizes the oracle can follow: the density Hessian and
the Pulay terms in several chunks, and the FP64 products with an item's points in two CTAs and in one (few items: four).
Bars as in the other parity tests: FP64 1e-12, FP32 1e-6, split 1e-10 of the magnitude sums."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

import oracle
from paper_1912_06636_gb300 import nao, synth
from tests._metrics import rel_err
from tests.test_gpu_edges import cuda, one_atom, shells

pytestmark = pytest.mark.gpu

TOL = {"fp64": 1e-12, "fp32": 1e-6, "split": 1e-10}


def pulay_close(got, ref, mag, tol):
    for c in range(3):
        assert np.max(np.abs(got[c] - ref[c])) <= tol * mag[c].max(), c


@pytest.mark.parametrize("n", [33, 65, 129])
def test_hessian_and_pulay_in_chunks(n):
    s = one_atom(shells(n), 240, seed=n)
    o = oracle.Oracle(s)
    v, P = s.potential(), synth.density_matrix(s, 2)
    nref, D, _ = o.density(s.pt_xyz, P, s.pt_w)
    gref, Dg = o.density_gradient(s.pt_xyz, P)
    href, Dh = o.density_hessian(s.pt_xyz, P)
    M, S, AM, AS = o.pulay_matrices(s.pt_xyz, s.pt_w, v)
    # room for one or two batches' ten rows (of at most 48 points): a chunk each
    with nao.Grid(s, device=0, max_batch_points=40, scratch_bytes=int(1.5 * n * 10 * 48 * 8)) as g:
        assert len(g.batches()[0]) - 1 >= 6
        for prec, tol in TOL.items():
            x, gr, h, _ = (t.cpu().numpy() for t in g.density_hessian(cuda(P), prec=prec))
            g.sync()
            assert rel_err(x, nref, D) <= tol, prec
            for c in range(3):
                assert rel_err(gr[c], gref[:, c], Dg[:, c]) <= tol, (prec, c)
            for k in range(6):
                assert rel_err(h[k], href[:, k], Dh[:, k]) <= tol, (prec, k)
            if prec != "split":
                m, x = (t.cpu().numpy() for t in g.pulay_matrices(cuda(v), prec=prec))
                pulay_close(m, M, AM, tol)
                pulay_close(x, S, AS, tol)


# (points of one batch, batches at least): with 129 functions a batch has 6 items of H and 9 of the Pulay terms; two CTAs
# per item from 1520 items on, one from 3040
@pytest.mark.parametrize("points,batches,h_items,p_items", [(620, 310, (1520, 3040), (1520, 3040)),
                                                           (1200, 600, (3040, 1 << 30), (3040, 1 << 30))])
def test_point_segments(points, batches, h_items, p_items):
    s = one_atom(shells(129), points, seed=points)
    o = oracle.Oracle(s)
    v = s.potential()
    H, A = o.hamiltonian(s.pt_xyz, s.pt_w, v)
    M, S, AM, AS = o.pulay_matrices(s.pt_xyz, s.pt_w, v)
    with nao.Grid(s, device=0, max_batch_points=2) as g:
        nb = len(g.batches()[0]) - 1
        assert nb >= batches and h_items[0] <= 6 * nb < h_items[1] and p_items[0] <= 9 * nb < p_items[1]
        h = g.integrate_h(cuda(v), prec="fp64").cpu().numpy()
        m, x = (t.cpu().numpy() for t in g.pulay_matrices(cuda(v), prec="fp64"))
    assert rel_err(h, H, A) <= TOL["fp64"]
    pulay_close(m, M, AM, TOL["fp64"])
    pulay_close(x, S, AS, TOL["fp64"])
