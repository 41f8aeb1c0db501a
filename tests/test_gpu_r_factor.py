"""R itself, and not only R^dag R: Householder's R has the phase -x_j / |x_j| on
row j, so its rows are fixed by the matrix, to eps ||x_j|| / |x_j| of the row."""

import numpy as np
import pytest

import paper_2605_29514_gb300 as stn

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

CDT = {0: torch.complex128, 1: torch.complex64}
EPS = {0: 2.2e-16, 1: 1.2e-7}


@pytest.fixture(scope="module", autouse=True)
def built():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    stn.build()


def graded(rng, m, n, precision):
    """Singular values over six decades, as the bonds of a state have."""
    k = min(m, n)
    u, v = (np.linalg.qr(rng.normal(size=(x, k)) + 1j * rng.normal(size=(x, k)))[0] for x in (m, n))
    return ((u * 10.0 ** (-6.0 * np.arange(k) / k)) @ v.conj().T).astype([np.complex128, np.complex64][precision])


def r_factor(precision, a):
    r = torch.tensor(a, device="cuda")
    stn.dense_qr(precision, *a.shape, r.data_ptr())
    return r.cpu().numpy()


@pytest.mark.parametrize("precision,m,n", [(1, 512, 250), (1, 512, 256), (1, 400, 200), (1, 300, 120), (1, 241, 512),
                                           (1, 480, 48), (1, 700, 300), (0, 200, 100), (0, 300, 49), (0, 130, 129)])
def test_cluster_has_the_r_of_one_cta(precision, m, n):
    """The R factor by a cluster's CTAs is that of one CTA (which the call with an
    explicit Q runs on), to the last bit."""
    a = graded(np.random.default_rng(m + n), m, n, precision)
    k = min(m, n)
    b, q, work = torch.tensor(a, device="cuda"), *(torch.zeros(m, k, dtype=CDT[precision], device="cuda") for _ in "qw")
    stn.dense_qr_q(precision, m, n, b.data_ptr(), q.data_ptr(), work.data_ptr())
    assert np.array_equal(r_factor(precision, a), b.cpu().numpy())


@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("m,n", [(1, 1), (5, 3), (40, 20), (70, 65), (100, 70), (150, 75), (300, 120), (512, 250)])
def test_rows_have_householder_phases(precision, m, n):
    """Rows against float64 reflections of the same matrix (Gaussian, at least
    as tall as wide, so of small condition): the rounding level of an R factor,
    64 eps sqrt(size) of the matrix norm, times ||x_j|| / |x_j| for row j."""
    rng = np.random.default_rng(m * n)
    a = (rng.normal(size=(m, n)) + 1j * rng.normal(size=(m, n))).astype([np.complex128, np.complex64][precision])
    r = r_factor(precision, a)
    ref, bound = a.astype(np.complex128), np.zeros(n)
    level = 64 * EPS[precision] * np.sqrt(m * n) * np.linalg.norm(ref)
    for j in range(n):
        x = ref[j:, j].copy()
        norm = np.linalg.norm(x)
        gamma = -x[0] / abs(x[0]) * norm
        bound[j] = level * norm / abs(x[0])
        x[0] -= gamma
        x /= np.linalg.norm(x)
        ref[j:, j:] -= 2 * np.outer(x, x.conj() @ ref[j:, j:])
        ref[j + 1:, j] = 0
    assert np.all(np.abs(r[:n] - ref[:n]).max(axis=1) < bound)


@pytest.mark.parametrize("m,n", [(5, 3), (40, 20), (60, 50), (100, 70), (140, 100), (160, 150)])
def test_r_without_q_is_r_with_q(m, n):
    """Complex64: the same R to the last bit with and without Q, at sizes whose
    columns fit shared memory with Q, without it only, or not at all."""
    a = graded(np.random.default_rng(m + n), m, n, 1)
    k = min(m, n)
    b, q, work = torch.tensor(a, device="cuda"), *(torch.zeros(m, k, dtype=CDT[1], device="cuda") for _ in "qw")
    stn.dense_qr_q(1, m, n, b.data_ptr(), q.data_ptr(), work.data_ptr())
    assert np.array_equal(r_factor(1, a), b.cpu().numpy())
