"""The large class (csrc/lsq_dense.cu) at the footprints where one block shape gives
way to the next: windows of few unknowns over rows that fill 70 to 110 KB, and all
shapes in one launch, against the oracle column by column, and through a plan, which
clears and reuses the lists between the launches."""
import numpy as np
import pytest
import scipy.sparse as sp

from paper_2406_17656_gb300 import workloads as W
from tests.test_gpu_dense_columns import _check, _window, sam  # noqa: F401

pytestmark = pytest.mark.gpu


def _rand(n, k, seed):
    """Two matrices of k random entries per column and a dominant diagonal."""
    rng = np.random.default_rng(seed)
    c, r = np.concatenate([rng.permutation(n) for _ in range(k)]), np.tile(np.arange(n), k)
    out = []
    for _ in range(2):
        m = sp.coo_matrix((rng.uniform(-1, 1, n * k), (r, c)), shape=(n, n)).tocsr()
        out.append(W.CSR.from_scipy((m + sp.diags(np.full(n, 2.0 * k))).tocsr()))
    return out


@pytest.mark.parametrize("n,k,nj", [(1100, 62, 14), (1500, 60, 14), (4000, 60, 14), (3000, 45, 20), (5000, 40, 22),
                                    (2000, 29, 27), (3000, 11, 40)])
def test_footprints(sam, n, k, nj):  # noqa: F811
    mats = _rand(n, k, n + nj)
    cp, ri = _window(n, nj)
    _check(sam, mats, cp, ri, 1)


def _mixed(n, seed):
    """Columns of 3 to 60 entries in blocks, so that every shape has some."""
    rng = np.random.default_rng(seed)
    k = np.repeat(rng.choice([3, 12, 30, 60], n // 25), 25)
    r = np.concatenate([rng.choice(n, c, replace=False) for c in k])
    c = np.repeat(np.arange(n), k)
    out = []
    for _ in range(2):
        m = sp.coo_matrix((rng.uniform(-1, 1, len(r)), (r, c)), shape=(n, n)).tocsr()
        out.append(W.CSR.from_scipy((m + sp.diags(np.full(n, 130.0))).tocsr()))
    return out


@pytest.mark.parametrize("steps", [1, 2, "auto"])
def test_every_shape_in_one_launch(sam, steps):  # noqa: F811
    mats = _mixed(2000, 5)
    cp, ri = _window(2000, 14)
    _check(sam, mats, cp, ri, steps)


@pytest.mark.parametrize("steps", [1, "auto"])
def test_plan_of_every_shape(sam, steps):  # noqa: F811
    import torch

    n = 4000
    mats = _mixed(n, 6)
    cp, ri = _window(n, 14)
    with sam.Handle() as h:
        A0, A1 = (sam.Csr.from_host(m) for m in mats)
        S = h.sam_pattern_from_csc(n, torch.from_numpy(cp).cuda(), torch.from_numpy(ri).cuda())
        one = h.sam_build(A1, A0, S, "fp32r", steps)
        plan = h.sam_plan_create([A1, A1], A0, [S, S], "fp32r", steps)
        plan.execute()
        plan.execute()
        h.sam_sync()
        assert torch.equal(plan.M_val, torch.cat([one[2]] * 2))
        plan.destroy()
        S.destroy()
