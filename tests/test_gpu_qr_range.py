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
