"""sam_residual's rows (csrc/residual_row.cuh) on both sides of the rule that
sums them through the ranks of their columns: 768 candidates, a span of
32,768 columns, rows out of order under SAM_FLAG_TRUSTED."""
import numpy as np
import pytest
import scipy.sparse as sp

from paper_2406_17656_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def sam():
    torch = pytest.importorskip("torch")
    from paper_2406_17656_gb300 import build, sam as S

    build.build()
    assert torch.cuda.is_available()
    return S


def _rows(rng, n, k, lo, hi):
    """k entries in each row at random columns of [lo, hi)."""
    cols = np.concatenate([np.sort(rng.choice(hi - lo, k, replace=False)) + lo for _ in range(n)])
    return sp.csr_matrix((rng.standard_normal(n * k), cols, np.arange(n + 1) * k), shape=(n, n))


def _bound(A, M, Z, fro):
    """A row sums at most 1024 products and its squares, a block sum of the
    rows follows: 2^11 roundings against the absolute values."""
    big = abs(A).dot(abs(M)) + abs(Z)
    return 2.0 ** 11 * 2.0 ** -53 * (np.sqrt(big.multiply(big).sum()) + fro)


def _check(sam, h, A, M, Z, dev=None):
    fro, rel = h.sam_residual(*(dev or [sam.Csr.from_host(W.CSR.from_scipy(x)) for x in (A, M, Z)]))
    R = (A.dot(M) - Z).tocsr()
    want, z = np.sqrt(R.multiply(R).sum()), np.sqrt(Z.multiply(Z).sum())
    tol = _bound(A, M, Z, want)
    assert abs(fro - want) <= tol
    assert abs(rel - want / z) <= 2 * tol / z


@pytest.mark.parametrize("ka,km,kz", [(1, 1, 1), (9, 25, 9), (23, 33, 9), (24, 32, 1), (40, 19, 7), (31, 33, 1)])
def test_rows_around_the_candidate_limit(sam, ka, km, kz):
    """Up to 768 candidates go through ranks, 769 to 1024 through the sort;
    (40, 19, 7): rows of A_k longer than a warp."""
    rng = np.random.default_rng(ka * km)
    n = 200
    A, M, Z = _rows(rng, n, ka, 0, n), _rows(rng, n, km, 0, n), _rows(rng, n, kz, 0, n)
    _check(sam, sam.Handle(), A, M, Z)


@pytest.mark.parametrize("last", [32766, 32767, 32768])
def test_rows_around_the_span_limit(sam, last):
    """Columns 0 and `last` of A_0 set the span; rows 1 and 2 are empty."""
    rng = np.random.default_rng(last)
    n = 32769
    keep = sp.diags(np.r_[1.0, 0.0, 0.0, np.ones(n - 3)])
    A = (keep @ sp.diags([rng.standard_normal(n), rng.standard_normal(n - 1)], [0, 1])).tocsr()
    M = sp.diags([rng.standard_normal(n), rng.standard_normal(n - 5)], [0, -5]).tocsr()
    z = np.setdiff1d(np.arange(0, n, 7), [1, 2])
    Z = sp.csr_matrix((rng.standard_normal(2 * len(z)), (np.repeat(z, 2), np.tile([0, last], len(z)))), shape=(n, n))
    A.eliminate_zeros()
    _check(sam, sam.Handle(), A, M, Z)


def test_rows_out_of_order_are_sorted(sam):
    """An unvalidated map with its rows reversed, and one with a column
    given twice: the values of the ordered one."""
    rng = np.random.default_rng(5)
    n = 100
    A, M, Z = (_rows(rng, n, k, 0, n) for k in (5, 6, 3))
    rev = W.CSR(n, M.indptr.astype(np.int32), M.indices.reshape(n, 6)[:, ::-1].ravel().astype(np.int32),
                M.data.reshape(n, 6)[:, ::-1].ravel().copy())
    twice = W.CSR(n, M.indptr.astype(np.int32), M.indices.copy().astype(np.int32), M.data.copy())
    twice.indices.reshape(n, 6)[:, 1] = twice.indices.reshape(n, 6)[:, 0]
    h = sam.Handle(trusted=True)
    dA, dZ = (sam.Csr.from_host(W.CSR.from_scipy(x)) for x in (A, Z))
    for m in (rev, twice):
        full = sp.coo_matrix((m.data, (np.repeat(np.arange(n), 6), m.indices)), shape=(n, n)).tocsr()
        _check(sam, h, A, full, Z, [dA, sam.Csr.from_host(m), dZ])
