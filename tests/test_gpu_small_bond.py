"""The routines of bonds that fit shared memory, at the sizes where they can go
wrong: the untiled contraction (one column, one row, row counts around the
rows in flight, the widest output), the shared-memory QR (columns around a
warp's four and the CTA's 64 groups, both sides of its capacity) and the
pivoted double-precision SVD (rank-deficient, zero and badly scaled matrices,
the column limit).  References are numpy in float64; bounds are rounding
levels: 64 eps sqrt(size) of the matrix norm."""

import numpy as np
import pytest

import paper_2605_29514_gb300 as stn

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

CDT = {0: torch.complex128, 1: torch.complex64}
RDT = {0: torch.float64, 1: torch.float32}
EPS = {0: 2.2e-16, 1: 1.2e-7}


@pytest.fixture(scope="module", autouse=True)
def built():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    stn.build()


def cmat(rng, m, n, precision):
    return (rng.normal(size=(m, n)) + 1j * rng.normal(size=(m, n))).astype([np.complex128, np.complex64][precision])


@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("op_a,op_b", [(0, 0), (0, 1), (1, 0), (1, 1)])
@pytest.mark.parametrize("m,n,k", [(1, 1, 1), (1, 511, 3), (2, 512, 5), (3, 513, 2), (512, 1, 7), (513, 1, 2),
                                   (9, 257, 4), (17, 31, 33), (32, 64, 32), (32, 64, 33)])
def test_untiled_contraction(precision, op_a, op_b, m, n, k):
    rng = np.random.default_rng(m + 100 * n + 7 * k)
    a = cmat(rng, *((k, m) if op_a else (m, k)), precision)
    b = cmat(rng, *((n, k) if op_b else (k, n)), precision)
    c0 = cmat(rng, m, n, precision)
    da, db, dc = (torch.tensor(x, device="cuda") for x in (a, b, c0))
    st = torch.zeros(1, dtype=torch.int32, device="cuda")
    stn.dense_cgemm(precision, op_a, op_b, m, n, k, da.data_ptr(), a.shape[1], db.data_ptr(), b.shape[1],
                    dc.data_ptr(), n, st.data_ptr(), alpha=0.5 - 0.25j, beta=-2.0)
    oa, ob = (x.astype(np.complex128) for x in (a, b))
    oa, ob = (oa.conj().T if op_a else oa), (ob.conj().T if op_b else ob)
    ref = (0.5 - 0.25j) * (oa @ ob) - 2.0 * c0
    scale = np.abs(oa) @ np.abs(ob) + 2.0 * np.abs(c0)
    assert (np.abs(dc.cpu().numpy() - ref) / scale).max() < 4 * (k + 4) * EPS[precision]


@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("m,n", [(1, 1), (1, 5), (5, 1), (2, 3), (3, 4), (4, 5), (16, 63), (70, 64), (70, 65), (66, 129),
                                 (91, 85), (91, 95), (200, 110)])
def test_shared_memory_qr(precision, m, n):
    """R^dag R = A^dag A with R upper trapezoidal, A = Q R with orthonormal Q."""
    rng = np.random.default_rng(31 * m + n)
    a = cmat(rng, m, n, precision)
    a[:, n // 2] = 0  # a zero column gets no reflector
    k = min(m, n)
    r = torch.tensor(a, device="cuda")
    stn.dense_qr(precision, m, n, r.data_ptr())
    b, q, work = torch.tensor(a, device="cuda"), torch.zeros(m, k, dtype=CDT[precision], device="cuda"), None
    work = torch.zeros(m, k, dtype=CDT[precision], device="cuda")
    stn.dense_qr_q(precision, m, n, b.data_ptr(), q.data_ptr(), work.data_ptr())
    a = a.astype(np.complex128)
    bound = 64 * EPS[precision] * np.sqrt(m * n) * np.linalg.norm(a)
    r, b, q = (x.cpu().numpy().astype(np.complex128) for x in (r, b, q))
    for x in (r, b):
        assert np.all(x[k:] == 0) and np.all(np.tril(x[:k, :k], -1) == 0)
        assert np.abs(x.conj().T @ x - a.conj().T @ a).max() <= bound * np.linalg.norm(a)
    assert np.abs(q @ b[:k] - a).max() <= bound
    assert np.abs(q.conj().T @ q - np.eye(k)).max() < 64 * EPS[precision] * np.sqrt(m * n)


@pytest.mark.parametrize("m,n,rank", [(1, 1, 1), (1, 9, 1), (9, 1, 1), (4, 4, 2), (7, 5, 5), (33, 64, 20), (64, 64, 64),
                                      (65, 64, 31), (40, 65, 40), (20, 128, 20), (20, 129, 20), (90, 90, 3)])
@pytest.mark.parametrize("scale", [1.0, 1e-60])
def test_pivoted_svd(m, n, rank, scale):
    """complex128: singular values and right vectors of matrices of full and
    deficient rank, with values over ten decades, and of a badly scaled one (not
    beyond 128 columns: the general path's QR takes columns below 1e-30 as zero)."""
    if n > 128 and scale != 1.0:
        pytest.skip("the general path treats columns below 1e-30 as zero")
    rng = np.random.default_rng(5 * m + n)
    u, _ = np.linalg.qr(cmat(rng, m, rank, 0))
    v, _ = np.linalg.qr(cmat(rng, n, rank, 0))
    s = scale * 10.0 ** (-10.0 * np.arange(rank) / rank)
    a = (u * s) @ v.conj().T
    da = torch.tensor(a, device="cuda")
    dv = torch.full((n, n), np.nan, dtype=torch.complex128, device="cuda")
    ds = torch.full((n,), np.nan, dtype=torch.float64, device="cuda")
    stn.dense_svd_noalloc(0, m, n, da.data_ptr(), dv.data_ptr(), ds.data_ptr())
    sig = np.sqrt(ds.cpu().numpy())
    vecs = dv.cpu().numpy()  # rows: columns of V
    order = np.argsort(-sig)
    bound = 64 * EPS[0] * np.sqrt(m * n)
    assert np.abs(sig[order[:rank]] - s).max() < bound * scale
    assert np.all(sig[order[rank:]] < bound * scale)
    vk = vecs[order[:rank]].T
    assert np.abs(vk.conj().T @ vk - np.eye(rank)).max() < bound
    assert np.abs(a @ vk @ vk.conj().T - a).max() < bound * scale
    assert np.all(np.isfinite(vecs))


def test_pivoted_svd_zero_and_non_finite():
    for value in (0.0, np.nan, np.inf):
        a = torch.zeros(6, 5, dtype=torch.complex128, device="cuda")
        a[3, 2] = value
        dv = torch.full((5, 5), 7.0, dtype=torch.complex128, device="cuda")
        ds = torch.full((5,), 7.0, dtype=torch.float64, device="cuda")
        stn.dense_svd_noalloc(0, 6, 5, a.data_ptr(), dv.data_ptr(), ds.data_ptr())
        if value == 0.0:
            assert torch.all(ds == 0) and torch.all(dv == 0)
        else:
            assert not torch.any(torch.isfinite(ds))


@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("cutoff,cap,theta,basis", [(1e-12, 64, 0.05, "Z"), (1e-12, 64, 0.0225, "X"), (5e-6, 64, 0.05, "X"),
                                                    (1e-3, 64, 0.05, "X"), (1e-3, 3, 0.1, "Z"), (5e-6, 1, 0.1, "X")])
def test_truncations_against_oracle(precision, cutoff, cap, theta, basis):
    """Truncations whose Jacobi ends without a sweep that finds nothing: full and
    capped ranks, cutoffs inside and below the spectrum.  Born probabilities and
    the largest bond against the oracle: rounding, 1e-9 in complex128 and 5e-5 in
    complex64 for states of a few hundred truncations."""
    if precision == 1 and cutoff < 5e-6:
        pytest.skip("below the rounding of complex64")
    from oracle.shot import make_program, run_shot
    from workloads import D3_EXACT, theta_table

    w = D3_EXACT.with_(rounds=1, p=0.0, theta=theta, memory_basis=basis, precision=precision, chi_cap=cap,
                       svd_cutoff=cutoff, degeneracy_tol=cutoff)
    sim = stn.Simulator(w, max_shots=3)
    angles = theta_table(w, sim.n_pairs)
    out = sim.sample_shots(3, 11, angles)
    prog = make_program(w)
    for s in range(3):
        ref = run_shot(w, 11 + s, angles, prog)
        assert list(out["bits"][s]) == list(ref.record)
        rb = np.array(ref.born)
        assert (np.abs(out["born"][s] - rb) / np.maximum(rb, 1e-4)).max() < (1e-9 if precision == 0 else 5e-5)
        if precision == 0:
            assert out["max_chi"][s] == ref.max_chi
    sim.close()


@pytest.mark.parametrize("precision,m,n", [(1, 480, 47), (1, 470, 48), (1, 160, 150), (1, 241, 512), (1, 512, 255),
                                           (0, 300, 49), (0, 101, 95), (0, 130, 129), (0, 64, 512)])
def test_large_matrices_over_a_cluster(precision, m, n):
    """R factors and SVDs on both sides of the column count and capacity from
    which the CTAs of a cluster share them, with odd numbers of 16-column blocks,
    ragged last blocks and wide matrices.  Bounds as above; a Jacobi vector of
    complex64 carries sqrt(rotations) roundings more (15 sweeps at most)."""
    rng = np.random.default_rng(13 * m + n)
    a = cmat(rng, m, n, precision)
    k = min(m, n)
    r = torch.tensor(a, device="cuda")
    stn.dense_qr(precision, m, n, r.data_ptr())
    da = torch.tensor(a, device="cuda")
    dv = torch.full((n, n), np.nan, dtype=CDT[precision], device="cuda")
    ds = torch.full((n,), np.nan, dtype=RDT[precision], device="cuda")
    a = a.astype(np.complex128)
    bound = 64 * EPS[precision] * np.sqrt(m * n) * np.linalg.norm(a)
    r = r.cpu().numpy().astype(np.complex128)
    assert np.all(r[k:] == 0) and np.all(np.tril(r[:k, :k], -1) == 0)
    assert np.abs(r.conj().T @ r - a.conj().T @ a).max() <= bound * np.linalg.norm(a)
    stn.dense_svd_noalloc(precision, m, n, da.data_ptr(), dv.data_ptr(), ds.data_ptr())
    sig = np.sqrt(ds.cpu().numpy().astype(np.float64))
    order = np.argsort(-sig)[:k]
    vk = dv.cpu().numpy()[order].T.astype(np.complex128)
    assert np.abs(sig[order] - np.linalg.svd(a, compute_uv=False)).max() < bound
    grow = np.sqrt(15 * k)
    assert np.abs(vk.conj().T @ vk - np.eye(k)).max() < 64 * EPS[precision] * np.sqrt(m * n) * grow
    assert np.abs(a @ vk @ vk.conj().T - a).max() < bound * grow


@pytest.mark.parametrize("precision,scales", [(1, (1.0, 1e-12, 1e12, 1e-25)), (1, (1e-20,)), (0, (1.0, 1e70, 1e-25)),
                                              (0, (1e75,))])
@pytest.mark.parametrize("m,n", [(3, 2), (40, 20), (100, 70), (128, 30), (129, 30), (400, 40)])
def test_qr_of_columns_far_from_one(precision, scales, m, n):
    """Columns whose reflectors are scaled by a power of two, beside ordinary
    ones; a Householder QR is backward stable column by column, so the bounds hold
    relative to each column's norm.  128 and 129 rows: both steps of the integer
    column norm."""
    rng = np.random.default_rng(m * n)
    size = np.array([scales[c % len(scales)] for c in range(n)])
    a = (cmat(rng, m, n, 0) * size).astype([np.complex128, np.complex64][precision])
    b, q = torch.tensor(a, device="cuda"), torch.zeros(m, n, dtype=CDT[precision], device="cuda")
    work = torch.zeros(m, n, dtype=CDT[precision], device="cuda")
    stn.dense_qr_q(precision, m, n, b.data_ptr(), q.data_ptr(), work.data_ptr())
    b, q = (x.cpu().numpy().astype(np.complex128) for x in (b, q))
    a = a.astype(np.complex128)
    bound = 64 * EPS[precision] * np.sqrt(m * n)
    assert np.abs(q.conj().T @ q - np.eye(n)).max() < bound
    assert (np.abs(q @ b[:n] - a).max(axis=0) / np.linalg.norm(a, axis=0)).max() < bound
