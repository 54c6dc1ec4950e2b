"""The Bloch sum against complex sums in numpy: an output array on any 8-byte boundary, images far from the origin,
cells of few functions with long lists of images."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_1912_06636_gb300 import nao

pytestmark = pytest.mark.gpu


def cuda(a):
    return torch.from_numpy(np.ascontiguousarray(a)).cuda()


def inputs(n_rs, nb, n_images, n_k, seed=9):
    rng = np.random.Generator(np.random.PCG64(seed))
    lat = np.array([[6.0, 0, 0], [0.8, 6.5, 0], [0, 0.5, 7.0]])
    return (rng.normal(size=(n_rs, n_rs)), rng.integers(0, nb, n_rs).astype(np.int32),
            rng.integers(0, n_images, n_rs).astype(np.int32), rng.integers(-2, 3, (n_images, 3)).astype(np.int32), lat,
            rng.uniform(-0.5, 0.5, (n_k, 3)))


def reference(h, fm, fi, cell, lat, k, nb):
    """(h(k), the sums of the terms' magnitudes)"""
    T = (cell.astype(np.float64) @ lat)[fi]
    F = np.zeros((len(k), len(fm), nb), complex)
    for q in range(len(k)):
        F[q, np.arange(len(fm)), fm] = np.exp(1j * (T @ k[q]))
    return (np.swapaxes(F.conj(), 1, 2) @ (h @ F), np.swapaxes(np.abs(F), 1, 2) @ (np.abs(h) @ np.abs(F)))


# 2000 images: their phases do not fit in shared memory, so the general form runs
@pytest.mark.parametrize("n_rs,nb,n_images,n_k", [(60, 7, 5, 8), (33, 5, 3, 1), (60, 7, 2000, 9)])
def test_output_on_an_odd_double(n_rs, nb, n_images, n_k):
    h, fm, fi, cell, lat, k = inputs(n_rs, nb, n_images, n_k)
    ref, A = reference(h, fm, fi, cell, lat, k, nb)
    n = 2 * n_k * nb * nb
    hk = torch.full((n + 2,), 7.0, dtype=torch.float64, device="cuda")
    at = hk.data_ptr() + 8
    assert at % 16 == 8
    d = [cuda(x) for x in (h, fm, fi, cell, k)]
    a9 = np.ascontiguousarray(lat.reshape(9))
    st = nao.load().nao_bloch_sum(d[0].data_ptr(), n_rs, d[1].data_ptr(), d[2].data_ptr(), d[3].data_ptr(), n_images,
                                  a9.ctypes.data, d[4].data_ptr(), n_k, nb, at, None, None)
    torch.cuda.synchronize()
    assert st == 0
    got = hk.cpu().numpy()
    assert got[0] == 7.0 and got[-1] == 7.0  # and nothing beside the array is written
    got = got[1:-1].reshape(n_k, nb, nb, 2)
    assert np.max(np.abs(got[..., 0] + 1j * got[..., 1] - ref)) <= 1e-13 * A.max()


@pytest.mark.parametrize("far", [0, 1000, -30000])
def test_images_far_from_the_origin(far):
    """h(k) depends on the images' differences alone: cells that all lie `far` lattice vectors away leave it as it is,
    to the rounding of a few hundred terms."""
    n_rs, nb, n_images, n_k = 120, 9, 6, 5
    h, fm, fi, cell, lat, k = inputs(n_rs, nb, n_images, n_k)
    ref, A = reference(h, fm, fi, cell, lat, k, nb)
    hk = nao.nao_bloch_sum(cuda(h), cuda(fm), cuda(fi), cuda(cell + np.int32(far)), lat, cuda(k), nb).cpu().numpy()
    assert np.max(np.abs(hk - ref) / A) <= 1e-14


# on both sides of 128 functions, up to which several threads share a column; lists of up to 500 images
@pytest.mark.parametrize("n_rs,nb,n_images,n_k", [(500, 1, 40, 3), (1600, 4, 400, 8), (1300, 13, 100, 1), (700, 100, 9, 4),
                                                 (640, 128, 5, 9), (645, 129, 5, 2)])
def test_small_cells(n_rs, nb, n_images, n_k):
    """The sums of a few hundred thousand terms at most, each rounded a few times, and the same twice."""
    h, fm, fi, cell, lat, k = inputs(n_rs, nb, n_images, n_k)
    ref, A = reference(h, fm, fi, cell, lat, k, nb)
    d = [cuda(x) for x in (h, fm, fi, cell)]
    hk, again = (nao.nao_bloch_sum(*d, lat, cuda(k), nb).cpu().numpy() for _ in range(2))
    assert np.max(np.abs(hk - ref) / A) <= 1e-13
    assert np.array_equal(hk, again)


# tables just below and just above the row form's shared memory, with 129 functions and with 128
@pytest.mark.parametrize("nb,kb", [(129, 226), (128, 222)])
@pytest.mark.parametrize("over", [0, 1])
def test_largest_tables(nb, kb, over):
    n_rs, n_k = 140, 8
    n_images = (kb * 1024 - 8 * (n_rs + nb + 1)) // 128 + over
    h, fm, fi, cell, lat, k = inputs(n_rs, nb, n_images, n_k)
    ref, A = reference(h, fm, fi, cell, lat, k, nb)
    hk = nao.nao_bloch_sum(cuda(h), cuda(fm), cuda(fi), cuda(cell), lat, cuda(k), nb).cpu().numpy()
    assert np.max(np.abs(hk - ref)) <= 1e-13 * A.max()
