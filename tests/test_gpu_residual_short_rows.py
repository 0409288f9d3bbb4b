"""sam_residual's rows (csrc/residual_row.cuh) at 32 and 33 candidates, where the
sort gives way to the columns' ranks, over short and wide spans, and both kinds
of row in one matrix."""
import numpy as np
import pytest
import scipy.sparse as sp

from tests.test_gpu_residual_rows import _check, _rows, sam  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [40, 3000, 30000])
@pytest.mark.parametrize("ka,km,kz", [(1, 31, 1), (4, 7, 3), (4, 7, 4), (4, 7, 5), (5, 6, 3), (31, 1, 2)])
def test_rows_around_a_warp_of_candidates(sam, n, ka, km, kz):  # noqa: F811
    rng = np.random.default_rng(n + 100 * ka + kz)
    _check(sam, sam.Handle(), _rows(rng, n, ka, 0, n), _rows(rng, n, km, 0, n), _rows(rng, n, kz, 0, n))


def test_short_and_long_rows_side_by_side(sam):  # noqa: F811
    rng = np.random.default_rng(9)
    n = 500
    k = rng.integers(1, 9, n)
    cols = np.concatenate([np.sort(rng.choice(n, c, replace=False)) for c in k])
    A = sp.csr_matrix((rng.standard_normal(len(cols)), cols, np.concatenate([[0], np.cumsum(k)])), shape=(n, n))
    _check(sam, sam.Handle(), A, _rows(rng, n, 6, 0, n), _rows(rng, n, 3, 0, n))
