"""R factors of matrices at the ends of the number range."""

import numpy as np
import pytest

import paper_2605_29514_gb300 as stn

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

CDT = {0: torch.complex128, 1: torch.complex64}
SHAPES = [(1, 1), (5, 1), (5, 3), (40, 20), (100, 70), (200, 1), (600, 60)]


@pytest.fixture(scope="module", autouse=True)
def built():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    stn.build()


@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("m,n", SHAPES)
@pytest.mark.parametrize("value", [np.inf, -np.inf, np.nan])
def test_non_finite_matrix_has_no_finite_r(precision, m, n, value):
    rng = np.random.default_rng(m + n)
    a = torch.tensor(rng.normal(size=(m, n)) + 1j * rng.normal(size=(m, n)), device="cuda").to(CDT[precision])
    torch.view_as_real(a)[m - 1, n // 2, m % 2] = value
    stn.dense_qr(precision, m, n, a.data_ptr())
    assert not torch.all(torch.isfinite(torch.view_as_real(a)))


@pytest.mark.parametrize("precision,scales", [(1, (1e8, 1e33)), (1, (1e34, 1.0, 1e-20)), (1, (1e17, 1e19)),
                                              (0, (1e60, 1e140)), (0, (1e120, 1e-24)), (0, (1e89, 1e92))])
@pytest.mark.parametrize("m,n", [(1, 2), (3, 2), (40, 20), (20, 40), (100, 70), (400, 60)])
def test_columns_that_would_overflow_together(precision, scales, m, n):
    """Columns whose products leave the range, beside each other: R^dag R and
    A = Q R column by column, relative to the columns' norms (64 eps sqrt(size),
    as for ordinary matrices)."""
    eps = {0: 2.2e-16, 1: 1.2e-7}[precision]
    rng = np.random.default_rng(m * n)
    size = np.array([scales[c % len(scales)] for c in range(n)])
    k = min(m, n)
    a = ((rng.normal(size=(m, n)) + 1j * rng.normal(size=(m, n))) * size).astype([np.complex128, np.complex64][precision])
    r = torch.tensor(a, device="cuda")
    stn.dense_qr(precision, m, n, r.data_ptr())
    b, q, work = torch.tensor(a, device="cuda"), *(torch.zeros(m, k, dtype=CDT[precision], device="cuda") for _ in "qw")
    stn.dense_qr_q(precision, m, n, b.data_ptr(), q.data_ptr(), work.data_ptr())
    r, b, q = (x.cpu().numpy().astype(np.complex128) for x in (r, b, q))
    unit = a.astype(np.complex128) / size
    bound = 64 * eps * np.sqrt(m * n)
    norm = np.linalg.norm(unit, axis=0)
    assert np.abs(q.conj().T @ q - np.eye(k)).max() < bound
    assert (np.abs(q @ (b[:k] / size) - unit).max(axis=0) / norm).max() < bound
    for x in (r / size, b / size):
        assert (np.abs(x.conj().T @ x - unit.conj().T @ unit) / np.outer(norm, norm)).max() < bound


@pytest.mark.parametrize("m,n", [(1, 2), (2, 5), (20, 41), (60, 130)])
def test_wide_columns_of_another_size(m, n):
    """Complex128: columns that get no reflector may have squares out of range."""
    rng = np.random.default_rng(m)
    size = np.where(np.arange(n) < m, 1e60, 1e250)
    unit = rng.normal(size=(m, n)) + 1j * rng.normal(size=(m, n))
    b = torch.tensor(unit * size, device="cuda")
    r, q, work = b.clone(), *(torch.zeros(m, m, dtype=CDT[0], device="cuda") for _ in "qw")
    stn.dense_qr(0, m, n, r.data_ptr())
    stn.dense_qr_q(0, m, n, b.data_ptr(), q.data_ptr(), work.data_ptr())
    bound = 64 * 2.2e-16 * np.sqrt(m * n) * np.linalg.norm(unit, axis=0)
    for x in (r, b):
        assert np.all(np.abs(q.cpu().numpy() @ (x.cpu().numpy() / size) - unit).max(axis=0) < bound)
