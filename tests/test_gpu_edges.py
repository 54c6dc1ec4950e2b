"""Sizes at which the kernels' tilings can go wrong, against the oracle at the bars of the other parity
tests (FP64 1e-12, FP32 1e-6, split 1e-10 of the magnitude sums, see tests/_metrics.py): reduced bases around
the 16-, 32-, 48- and 64-function blocks, batches around the 16-, 32-, 64- and 128-point tiles, every angular
momentum up to 6 (the evaluation kernels are instantiated by the largest one), and both forms of the Bloch sum."""
import math

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


def shells(n):
    """Angular momenta whose functions number exactly n (f, d and p functions, the rest s)."""
    ls = []
    for l in (3, 2, 1, 0):
        while n >= 2 * l + 1 and (l == 0 or len(ls) % 4 != 3 or n > 40):
            ls.append(l)
            n -= 2 * l + 1
            if l and len(ls) % 5 == 4:
                break
    ls += [0] * n
    return ls


def one_atom(ls, n_points, seed=5):
    """One atom with the given functions and n_points random points inside every cutoff (so that each batch
    has all functions)."""
    rng = np.random.Generator(np.random.PCG64(seed))
    sp = synth.Species(ls=list(ls), alphas=list(np.exp(rng.uniform(math.log(0.2), math.log(3.0), len(ls)))), Z=6.0)
    s = synth.make_system([[0.1, -0.2, 0.3]], [0], [sp], n_rad=1, n_theta=1, n_phi=1)
    d = rng.normal(size=(n_points, 3))
    d *= (rng.uniform(0.15, 4.0, n_points) / np.linalg.norm(d, axis=1))[:, None]
    s.pt_xyz = np.ascontiguousarray(s.atom_xyz[0] + d)
    s.pt_w = rng.uniform(0.001, 0.01, n_points)
    return s


def check(s, B, precs=("fp64", "fp32", "split"), grad=False, tol=TOL, **opts):
    o = oracle.Oracle(s)
    v = s.potential()
    v[::3] *= -1.0  # both signs of the weights
    P = synth.density_matrix(s, 1)
    H, A = o.hamiltonian(s.pt_xyz, s.pt_w, v)
    n, D, ne = o.density(s.pt_xyz, P, s.pt_w)
    if grad:
        gref, Dg = o.density_gradient(s.pt_xyz, P)
    with nao.Grid(s, device=0, max_batch_points=B, **opts) as g:
        for prec in precs:
            h = torch.full((g.nb, g.nb), float("nan"), dtype=torch.float64, device="cuda")
            h = g.integrate_h(cuda(v), prec=prec, H=h).cpu().numpy()
            x, e = g.update_density(cuda(P), prec=prec)
            torch.cuda.synchronize()
            g.sync()
            assert rel_err(h, H, A) <= tol[prec], prec
            assert rel_err(x.cpu().numpy(), n, D) <= tol[prec], prec
            assert abs(float(e.item()) - ne) <= tol[prec] * float(np.sum(s.pt_w * D))
            if grad:
                _, gr, _ = g.density_gradient(cuda(P), prec=prec)
                for c in range(3):
                    assert rel_err(gr[c].cpu().numpy(), gref[:, c], Dg[:, c]) <= tol[prec], prec


@pytest.mark.parametrize("n", [1, 15, 16, 17, 31, 32, 33, 48, 49, 64, 65, 97, 129, 161])
def test_function_counts(n):
    s = one_atom(shells(n), 90)
    assert s.n_basis == n
    check(s, 45, grad=n in (17, 65))
    if n in (33, 65, 161):
        # 48-wide tiles; 10 slices carry 60 bits, and these batches span every function's whole range (the
        # header's figure for such batches is 1.6e-9)
        check(s, 45, precs=("split",), tol={"split": 1e-8}, split_slices=10, autotune=0)
        check(s, 45, precs=("split",), split_digits=1, split_slices=14)  # e4m3 digits
        check(s, 45, precs=("split",), split_digits=1, split_slices=15)  # and an odd number of slices


@pytest.mark.parametrize("B", [1, 15, 16, 17, 32, 33, 63, 64, 65, 127, 129, 300])
def test_batch_sizes(B):
    check(one_atom([0, 1, 2, 3, 0, 1], max(2 * B, 7), seed=B), B, grad=B in (17, 65))


@pytest.mark.parametrize("ls", [[0], [1, 0], [2, 1, 0], [3, 0, 2], [4, 4, 0, 1], [5, 0, 2], [6, 1, 0, 3]])
def test_angular_momenta(ls):
    s = one_atom(ls, 150, seed=sum(ls))
    check(s, 70, grad=True)
    o = oracle.Oracle(s)
    P = synth.density_matrix(s, 2)
    href, Dh = o.density_hessian(s.pt_xyz, P)
    v = s.potential()
    M, S, AM, AS = o.pulay_matrices(s.pt_xyz, s.pt_w, v)
    with nao.Grid(s, device=0, max_batch_points=70) as g:
        for prec in ("fp64", "fp32", "split"):
            hess = g.density_hessian(cuda(P), prec=prec)[2].cpu().numpy()
            g.sync()
            for k in range(6):
                assert rel_err(hess[k], href[:, k], Dh[:, k]) <= TOL[prec], (prec, k)
        for prec, scale in (("fp64", 1e-14), ("fp32", 1e-6)):  # at the matrices' scale, as the Pulay tests
            m, x = (t.cpu().numpy() for t in g.pulay_matrices(cuda(v), prec=prec))
            for c in range(3):
                assert np.max(np.abs(m[c] - M[c])) <= scale * AM[c].max() and np.max(np.abs(x[c] - S[c])) <= scale * AS[c].max()


def bloch_inputs(n_rs, nb, n_images, n_k, seed=3):
    rng = np.random.Generator(np.random.PCG64(seed))
    h = rng.normal(size=(n_rs, n_rs))
    h[rng.random((n_rs, n_rs)) < 0.4] = 0.0
    cell = rng.integers(-2, 3, size=(n_images, 3)).astype(np.int32)
    lat = np.array([[6.0, 0, 0], [0.8, 6.5, 0], [0, 0.5, 7.0]])
    return (h, rng.integers(0, nb, n_rs).astype(np.int32), rng.integers(0, n_images, n_rs).astype(np.int32), cell, lat,
            rng.uniform(-0.5, 0.5, (n_k, 3)))


def bloch_reference(h, fm, fi, cell, lat, k, nb):
    T = (cell.astype(np.float64) @ lat)[fi]
    F = np.zeros((len(k), len(fm), nb), complex)
    for q in range(len(k)):
        F[q, np.arange(len(fm)), fm] = np.exp(1j * (T @ k[q]))
    def fold(G, x):
        return np.swapaxes(G.conj(), 1, 2) @ (x @ G)

    return fold(F, h), fold(np.abs(F), np.abs(h))


# 2000 images: their phases for eight k points do not fit in shared memory, so the general form runs
@pytest.mark.parametrize("n_rs,nb,n_images,n_k", [(1, 1, 1, 1), (37, 5, 3, 2), (70, 7, 9, 3), (300, 260, 11, 8), (64, 9, 20, 17),
                                                 (50, 6, 2000, 9)])
def test_bloch_sum_forms(n_rs, nb, n_images, n_k):
    h, fm, fi, cell, lat, k = bloch_inputs(n_rs, nb, n_images, n_k)
    ref, A = bloch_reference(h, fm, fi, cell, lat, k, nb)
    err = torch.full((1,), -1, dtype=torch.int32, device="cuda")
    out = torch.full((n_k, nb, nb, 2), float("nan"), dtype=torch.float64, device="cuda")
    hk = nao.nao_bloch_sum(cuda(h), cuda(fm), cuda(fi), cuda(cell), lat, cuda(k), nb, out=out, err=err).cpu().numpy()
    assert int(err.item()) == 0
    assert np.max(np.abs(hk - ref)) <= 1e-13 * max(A.max(), 1.0)


@pytest.mark.parametrize("n_images", [4, 2000])
def test_bloch_sum_skips_and_counts_bad_entries(n_images):
    n_rs, nb, n_k = 40, 6, 8
    h, fm, fi, cell, lat, k = bloch_inputs(n_rs, nb, n_images, n_k)
    fm[3], fm[11], fi[20] = -1, nb, n_images
    bad = np.zeros(n_rs, bool)
    bad[[3, 11, 20]] = True
    hg = h.copy()
    hg[bad, :] = 0.0
    hg[:, bad] = 0.0
    ref, A = bloch_reference(hg, np.where(bad, 0, fm), np.where(bad, 0, fi), cell, lat, k, nb)
    hd, fmd, fid, cd, kd = cuda(h), cuda(fm), cuda(fi), cuda(cell), cuda(k)
    hk = torch.empty((n_k, nb, nb, 2), dtype=torch.float64, device="cuda")
    err = torch.zeros(1, dtype=torch.int32, device="cuda")
    A9 = np.ascontiguousarray(lat.reshape(9))
    st = nao.load().nao_bloch_sum(hd.data_ptr(), n_rs, fmd.data_ptr(), fid.data_ptr(), cd.data_ptr(), n_images, A9.ctypes.data,
                                  kd.data_ptr(), n_k, nb, hk.data_ptr(), err.data_ptr(), None)
    torch.cuda.synchronize()
    assert st == 0
    assert int(err.item()) == int(np.count_nonzero(h[bad | np.zeros(n_rs, bool)][:, :]) + np.count_nonzero(h[~bad][:, bad]))
    got = torch.view_as_complex(hk).cpu().numpy()
    assert np.max(np.abs(got - ref)) <= 1e-13 * max(A.max(), 1.0)
