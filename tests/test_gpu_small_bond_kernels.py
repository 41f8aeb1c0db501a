"""The routines of small bonds alone, for both CTA sizes: the SVD of the
truncation in double precision and in pairs of floats, with its matrix in shared
and in global memory; the QR; the keep rule; the contraction by one CTA; the roots and reciprocals.
References are numpy in float64.

Bounds: 64 eps sqrt(m n) of the working precision (1.1e-16; 1.4e-14 for pairs of
floats, 2^-46) relative to the matrix norm, and for results stored in single
precision 8 of its roundings of 6e-8 on top (a vector's components are rounded
one by one, which changes a product of two by two of them at most)."""

import ctypes
import os
import subprocess
from concurrent.futures import ThreadPoolExecutor

import numpy as np
import pytest

from paper_2605_29514_gb300 import _native

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

HERE = os.path.dirname(os.path.abspath(__file__))
CDT = {0: torch.complex128, 1: torch.complex64}
RDT = {0: torch.float64, 1: torch.float32}
NP = {0: np.complex128, 1: np.complex64}
EPS = {0: 1.1e-16, 1: 1.4e-14}
STORE = {0: 0.0, 1: 8 * 6e-8}


@pytest.fixture(scope="module")
def libs(tmp_path_factory):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    out = tmp_path_factory.mktemp("small_bond")

    def compiled(threads):
        so = str(out / f"checks{threads}.so")
        subprocess.run([_native.NVCC, *_native.ARCH, "-O3", "-std=c++17", f"-DSTN_CTA_THREADS={threads}", "-I",
                        _native.CSRC, "-I", _native.INCLUDE, "-Xcompiler", "-fPIC", "-shared",
                        os.path.join(HERE, "small_bond_checks.cu"), "-o", so], check=True, capture_output=True, text=True)
        return threads, ctypes.CDLL(so)

    with ThreadPoolExecutor() as ex:
        return dict(ex.map(compiled, (256, 512)))


def ptr(t):
    return ctypes.c_void_p(0 if t is None else t.data_ptr())


def svd(lib, precision, shared, a, cutoff=0.0, kmax=None):
    """lam, V (columns) and the rank; with kmax the truncation's: lam, the kept
    vectors, the site, keep and the discarded weight."""
    m, n = a.shape
    da = torch.tensor(a, device="cuda")
    lam = torch.full((n,), 7.0, dtype=RDT[precision], device="cuda")
    v, vs, site = (torch.full((n, n), 7.0, dtype=CDT[precision], device="cuda") for _ in range(3))
    work = torch.zeros(m * n, dtype=torch.complex128, device="cuda")
    out = torch.zeros(2, dtype=torch.int32, device="cuda")
    disc = torch.zeros(1, dtype=torch.float64, device="cuda")
    st = lib.check_svd(precision, int(shared), m, n, ptr(da), ptr(v), ptr(lam), ctypes.c_double(cutoff), kmax or 0,
                       ptr(work), ptr(vs), ptr(site), ptr(out), ptr(disc), int(kmax is not None))
    assert st == 0
    got, fail = out.cpu().numpy()
    lam = lam.cpu().numpy().astype(np.float64)
    if kmax is None:
        return lam, v.cpu().numpy().astype(np.complex128).reshape(n, n)[:got].T, got
    vectors = vs.reshape(-1)[: n * got].reshape(n, got).cpu().numpy().astype(np.complex128)
    return lam, vectors, site.reshape(-1)[: n * got].reshape(got, n).cpu().numpy(), got, disc.item(), fail


def low_rank(rng, m, n, rank, precision):
    """Small integers, so that the rank is exact in either precision (never 0)."""
    def part(*shape):
        return rng.integers(1, 4, shape) * (1 + 0j) + 1j * rng.integers(-3, 4, shape)

    return (part(m, rank) @ part(rank, n)).astype(NP[precision])


def graded(rng, m, n, precision, decades):
    k = min(m, n)
    u, v = (np.linalg.qr(rng.normal(size=(x, k)) + 1j * rng.normal(size=(x, k)))[0] for x in (m, n))
    return ((u * 10.0 ** (-decades * np.arange(k) / k)) @ v.conj().T).astype(NP[precision])


SIZES = [(1, 1), (1, 9), (9, 1), (5, 4), (16, 16), (30, 31), (33, 64), (64, 33), (64, 64), (65, 67), (100, 100), (104, 128),
         (40, 128)]


def check(a, lam, v, precision):
    m, n = a.shape
    a = a.astype(np.complex128)
    bound = 64 * EPS[precision] * np.sqrt(m * n) + STORE[precision]
    assert np.abs(v.conj().T @ v - np.eye(v.shape[1])).max() < bound
    sigma = np.zeros(n)
    sigma[: min(m, n)] = np.linalg.svd(a, compute_uv=False)
    assert np.abs(np.sort(np.sqrt(lam))[::-1] - sigma).max() <= bound * sigma[0]
    assert np.linalg.norm(a @ v @ v.conj().T - a, 2) <= 2 * bound * sigma[0]


@pytest.mark.parametrize("threads", [256, 512])
@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("shared", [True, False])
@pytest.mark.parametrize("m,n", SIZES)
@pytest.mark.parametrize("kind,scale", [("graded", 1.0), ("graded", 1e-10), ("low", 1.0), ("low", 2.0 ** 40)])
def test_svd(libs, threads, precision, shared, m, n, kind, scale):
    """Values and vectors, and at cutoff 0 the truncation's: every value counts,
    and nothing beyond the rank is kept."""
    if shared and 16 * n * (m | 1) > 220 * 1024:
        pytest.skip("larger than shared memory")
    rng = np.random.default_rng(7 * m + n)
    rank = max(1, min(m, n) // 3)
    a = (low_rank(rng, m, n, rank, precision) if kind == "low" else graded(rng, m, n, precision, 6.0)) * NP[precision](scale)
    lam, v, got = svd(libs[threads], precision, shared, a)
    check(a, lam, v[:, lam[:got] > 0], precision)
    lam, v, site, keep, disc, fail = svd(libs[threads], precision, shared, a, kmax=n)
    assert fail == 0 and 1 <= keep <= min(m, n) and disc < 1e-20
    check(a, lam, v, precision)
    if precision == 1:
        assert np.array_equal(site.astype(np.complex128), v.conj().T)


@pytest.mark.parametrize("threads", [256, 512])
@pytest.mark.parametrize("precision,cutoff", [(0, 1e-3), (0, 1e-9), (1, 1e-3), (1, 5e-6)])
@pytest.mark.parametrize("m,n", [(6, 4), (33, 64), (64, 64), (90, 100)])
def test_truncation(libs, threads, precision, cutoff, m, n):
    """The kept count, and the weight of the values that the cutoff or the cap drops."""
    a = graded(np.random.default_rng(m + n), m, n, precision, 5.3)
    sigma = np.linalg.svd(a.astype(np.complex128), compute_uv=False)
    count = int(np.sum(sigma > cutoff * sigma[0]))
    near = np.abs(sigma / (cutoff * sigma[0]) - 1).min()
    assert near > 1e-3  # no value at the cutoff
    for kmax in (n, max(1, count // 2)):
        _, v, _, keep, disc, fail = svd(libs[threads], precision, False, a, cutoff, kmax)
        assert fail == 0 and keep == min(count, kmax)
        drop = np.sum(sigma[keep:] ** 2) / np.sum(sigma ** 2)
        level = 64 * EPS[precision] * np.sqrt(m * n) + STORE[precision]
        assert abs(disc - drop) <= level * (np.sqrt(drop) + level)
        ref = np.linalg.svd(a.astype(np.complex128))[2][:keep].conj().T
        gap = sigma[keep - 1] - (sigma[keep] if keep < len(sigma) else 0.0)
        assert np.linalg.norm(ref - v @ (v.conj().T @ ref), 2) <= 4 * level * sigma[0] / gap + np.sqrt(level)


@pytest.mark.parametrize("threads", [256, 512])
@pytest.mark.parametrize("precision,small", [(0, 1e-12), (1, 1e-8)])
@pytest.mark.parametrize("kept,m,n", [(1, 8, 6), (4, 24, 20), (20, 60, 50)])
def test_weight_of_the_remainder(libs, threads, precision, small, kept, m, n):
    """An identity beside a block so small that the QR stops before it: its weight
    is the block's squared norm, to the rounding of the stored norms (1e-5)."""
    rng = np.random.default_rng(kept)
    a = np.zeros((m, n), dtype=NP[precision])
    a[:kept, :kept] = np.eye(kept)
    block = rng.normal(size=(m - kept, 1)) * rng.normal(size=(1, n - kept)) * small  # columns of unlike norms
    a[kept:, kept:] = block
    weight = np.linalg.norm(a[kept:, kept:].astype(np.complex128)) ** 2
    _, _, _, keep, disc, fail = svd(libs[threads], precision, True, a, 1e-3, n)
    assert fail == 0 and keep == kept
    assert disc == pytest.approx(weight / (kept + weight), rel=1e-5, abs=0)


@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("m,n", [(2, 2), (8, 4), (20, 16), (128, 128)])
def test_first_of_equal_columns_is_kept(libs, precision, m, n):
    """A cap that cuts a cluster of orthogonal columns of equal norm keeps the first."""
    a = np.zeros((m, n), dtype=NP[precision])
    a[np.arange(n) * (m // n), np.arange(n)] = 0.5j
    _, v, _, keep, _, fail = svd(libs[256], precision, False, a, 1e-6, 1)
    assert fail == 0 and keep == 1
    assert np.array_equal(np.abs(v[:, 0]), np.eye(n)[0])


@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("delta", [0.0, 1e-3])
def test_keep_count(libs, precision, delta):
    """The keep rule on squared values: those above the cutoff, and at most the cap
    of them that exceed the first dropped one by more than delta sigma_1.  Of equal
    values on both sides of the cap none is kept, whatever their size."""
    rng = np.random.default_rng(3)
    for trial in range(200):
        s = rng.uniform(0.1, 0.9)
        lam = np.array([1.0, s, s, s, s * s, 1e-12] + [0.0] * (trial % 60)).astype([np.float64, np.float32][precision])
        dl, out = torch.tensor(lam, device="cuda"), torch.zeros(1, dtype=torch.int32, device="cuda")
        perm = torch.arange(len(lam), dtype=torch.int32, device="cuda")
        for cap, want in ((1, 1), (2, 1), (3, 1), (4, 4), (5, 5), (6, 5), (len(lam) + 1, 5)):
            assert libs[512].check_keep(precision, ptr(dl), ptr(perm), len(lam), cap, ctypes.c_double(1e-5),
                                        ctypes.c_double(delta), ptr(out)) == 0
            assert out.item() == want


@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("shared", [True, False])
@pytest.mark.parametrize("value", [0.0, np.inf, np.nan])
def test_zero_and_non_finite(libs, precision, shared, value):
    a = np.zeros((7, 6), dtype=NP[precision])
    a[2, 3] = value
    lam, _, _ = svd(libs[256], precision, shared, a)
    _, v, _, keep, disc, fail = svd(libs[256], precision, shared, a, 1e-6, 6)
    if value == 0.0:
        assert np.all(lam == 0) and keep == 1 and fail == 0 and disc == 0
        assert np.array_equal(v[:, 0], np.eye(6)[0])
    else:
        assert not np.any(np.isfinite(lam)) and fail != 0


@pytest.mark.parametrize("threads", [256, 512])
@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("conj_t", [False, True])
@pytest.mark.parametrize("m,n", [(1, 1), (1, 5), (5, 1), (2, 3), (4, 5), (16, 63), (40, 20), (66, 64), (63, 65), (128, 30),
                                 (129, 30), (60, 70), (2, 400)])
@pytest.mark.parametrize("scales", [(1.0,), (1.0, 1e-12, 1e12, 1e-25)])
def test_qr(libs, threads, precision, conj_t, m, n, scales):
    """R and Q of the shared-memory QR, of the matrix or its conjugate transpose as
    stored, with a zero column and with columns far from one: relative to the
    columns' norms, 64 roundings of the precision times sqrt(size)."""
    rng = np.random.default_rng(31 * m + n)
    size = np.array([scales[c % len(scales)] for c in range(n)])
    a = ((rng.normal(size=(m, n)) + 1j * rng.normal(size=(m, n))) * size).astype(NP[precision])
    a[:, n // 2] = 0
    k = min(m, n)
    given = torch.tensor(np.ascontiguousarray(a.conj().T) if conj_t else a, device="cuda")
    r, r2 = (torch.full((k, n), 7.0, dtype=CDT[precision], device="cuda") for _ in range(2))
    q = torch.full((k, m) if conj_t else (m, k), 7.0, dtype=CDT[precision], device="cuda")
    assert libs[threads].check_qr(precision, int(conj_t), m, n, ptr(given), ptr(r), ptr(q)) == 0
    assert libs[threads].check_qr(precision, int(conj_t), m, n, ptr(given), ptr(r2), None) == 0
    assert torch.equal(r, r2)
    r, q = (x.cpu().numpy().astype(np.complex128) for x in (r, q))
    q = q.conj().T if conj_t else q
    unit = a.astype(np.complex128) / size
    norm = np.maximum(np.linalg.norm(unit, axis=0), 1e-3)
    bound = 64 * (1.1e-16 if precision == 0 else 6e-8) * np.sqrt(m * n)
    assert np.all(np.tril(r, -1) == 0)
    assert np.abs(q.conj().T @ q - np.eye(k)).max() < bound
    assert (np.abs(q @ (r / size) - unit).max(axis=0) / norm).max() < bound


@pytest.mark.parametrize("threads", [256, 512])
@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("op_a,op_b", [(0, 0), (0, 1), (1, 0)])
@pytest.mark.parametrize("m,n,k", [(1, 511, 3), (2, 512, 5), (3, 513, 2), (9, 257, 4), (1, 256, 7), (700, 1, 2), (17, 31, 33),
                                   (64, 64, 64), (65, 70, 40), (129, 130, 9), (200, 33, 66)])
def test_contraction_of_one_cta(libs, threads, precision, op_a, op_b, m, n, k):
    """Untiled and tiled products of a CTA: the widest rows, several blocks of rows,
    both tile heights with remainders.  k + 2 roundings of sums of |a||b|, twice."""
    rng = np.random.default_rng(m + 3 * n + 5 * k)
    a = (rng.normal(size=(k, m) if op_a else (m, k)) + 1j * rng.normal(size=(k, m) if op_a else (m, k))).astype(NP[precision])
    b = (rng.normal(size=(n, k) if op_b else (k, n)) + 1j * rng.normal(size=(n, k) if op_b else (k, n))).astype(NP[precision])
    da, db = torch.tensor(a, device="cuda"), torch.tensor(b, device="cuda")
    c = torch.full((m, n), 7.0, dtype=CDT[precision], device="cuda")
    assert libs[threads].check_gemm(precision, op_a, op_b, m, n, k, ptr(da), ptr(db), ptr(c)) == 0
    a, b = (x.astype(np.complex128) for x in (a, b))
    a, b = (a.conj().T if op_a else a), (b.conj().T if op_b else b)
    scale = np.abs(a) @ np.abs(b)
    assert (np.abs(c.cpu().numpy() - a @ b) / scale).max() < 4 * (k + 2) * (1.1e-16 if precision == 0 else 6e-8)


@pytest.mark.parametrize("what,decades,bound", [(0, 290, 3e-16), (1, 290, 2.3e-16), (2, 30, 2.0 ** -45), (3, 30, 2.0 ** -23)])
def test_roots_and_reciprocals(libs, what, decades, bound):
    """1 / sqrt(x) (0: double, 2: pairs of floats) and 1 / x (1: double, 3: pairs
    of floats, result in single precision) over the range of the exponents.  The
    starting value is good to 2^-20; a third-order step leaves the cube of that and
    the roundings of the step: one and a half of double's, a few of 2^-48 for
    pairs.  The single-precision reciprocal takes a second-order step: 2^-40 and a
    rounding, at most one unit in the last place."""
    rng = np.random.default_rng(what)
    x = np.concatenate([10.0 ** rng.uniform(-decades, decades, 20000), rng.uniform(1, 4, 20000), 2.0 ** np.arange(-40, 41)])
    if what >= 2:  # what a pair of floats holds
        h = x.astype(np.float32)
        x = h.astype(np.float64) + (x - h).astype(np.float32)
    dx, dy = torch.tensor(x, device="cuda"), torch.zeros(len(x), dtype=torch.float64, device="cuda")
    assert libs[512].check_math(what, len(x), ptr(dx), ptr(dy)) == 0
    wide = x.astype(np.longdouble)
    ref = 1 / np.sqrt(wide) if what in (0, 2) else 1 / wide
    assert np.abs(dy.cpu().numpy() / ref - 1).max() < bound


@pytest.mark.parametrize("pairs,decades,bound", [(0, 120, 16 * 1.1e-16), (1, 13, 2.0 ** -42)])
def test_reflector_heads(libs, pairs, decades, bound):
    """v0, gamma and beta of a column from its first element and squared norm, over
    norms of many decades; sixteen roundings of the working precision (2^-46 for
    pairs).  A first element of zero takes the phase 1."""
    rng = np.random.default_rng(pairs)
    count = 4000
    size = 10.0 ** rng.uniform(-decades, decades, count)
    share = rng.uniform(0.01, 1.0, count)  # |x_j| / ||x||
    phase = np.exp(2j * np.pi * rng.uniform(size=count))
    al = size * share * phase
    al[:5] = 0
    x = np.stack([al.real, al.imag, size ** 2], axis=1)
    if pairs:
        h = x.astype(np.float32)
        x = h.astype(np.float64) + (x - h).astype(np.float32)
    dx, dy = torch.tensor(x, device="cuda"), torch.zeros(count, 5, dtype=torch.float64, device="cuda")
    assert libs[512].check_heads(pairs, count, ptr(dx), ptr(dy)) == 0
    y = dy.cpu().numpy()
    re, im, norm2 = x.astype(np.longdouble).T
    norm, a = np.sqrt(norm2), np.sqrt(re * re + im * im)
    one = a == 0
    gr, gi = -np.where(one, norm, re / np.where(one, 1, a) * norm), -np.where(one, 0, im / np.where(one, 1, a) * norm)
    for got, want in ((y[:, 0], re - gr), (y[:, 1], im - gi), (y[:, 2], gr), (y[:, 3], gi)):
        assert (np.abs(got - want) / norm).max() < 2 * bound
    assert np.abs(y[:, 4] * norm * (norm + a) - 1).max() < bound
