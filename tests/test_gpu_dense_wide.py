"""The large class of refined FP32 builds (csrc/lsq_dense.cu) on columns whose rows
span more than 32,768: a mesh in a random numbering, 27-point stencils around that
span, and dense columns spread over 1.5 million rows.  Against the oracle column by
column, and none of them by the FP64 re-solve."""
import itertools

import numpy as np
import pytest
import scipy.sparse as sp

import oracle
from paper_2406_17656_gb300 import workloads as W
from tests import colcheck
from tests.test_gpu_dense_columns import _spread, sam  # noqa: F401

pytestmark = pytest.mark.gpu


def _stencil27(nx, ny, nz, seed):
    """Two matrices on the 27-point stencil of an nx x ny x nz grid."""
    idx = np.arange(nx * ny * nz).reshape(nz, ny, nx)
    rows, cols = [], []
    for o in itertools.product((-1, 0, 1), repeat=3):
        a = idx[tuple(slice(max(0, -d), s - max(0, d)) for d, s in zip(o, idx.shape))]
        b = idx[tuple(slice(max(0, d), s + min(0, d)) for d, s in zip(o, idx.shape))]
        rows.append(a.ravel())
        cols.append(b.ravel())
    r, c = np.concatenate(rows), np.concatenate(cols)
    rng = np.random.default_rng(seed)
    return [sp.csr_matrix((np.where(r == c, 30.0, rng.uniform(-1, 0, len(r))), (r, c)), shape=(idx.size, idx.size))
            for _ in range(2)]


def _some(cp, ri, n, cols):
    """The pattern with the columns `cols` of (cp, ri) and the diagonal elsewhere."""
    lists = [ri[cp[j]:cp[j + 1]] if j in cols else [j] for j in range(n)]
    return np.concatenate([[0], np.cumsum([len(x) for x in lists])]).astype(np.int32), np.concatenate(lists).astype(np.int32)


def _check(sam, mats, cp, ri, steps):  # noqa: F811
    import torch

    a0, a1 = mats
    n = a0.n
    with sam.Handle() as h:
        S = h.sam_pattern_from_csc(n, torch.from_numpy(cp).cuda(), torch.from_numpy(ri).cuda())
        r2 = torch.empty(n, dtype=torch.float64, device="cuda")
        rp, ci, v = h.sam_build(sam.Csr.from_host(a1), sam.Csr.from_host(a0), S, "fp32r", steps, res2=r2)
        h.sam_sync()
        stats = h.sam_refine_stats()
        S.destroy()
    assert stats[2] == 0
    ref = oracle.build(a1, a0, cp, ri)
    got = colcheck.csr_to_csc_values(n, rp.cpu().numpy(), ci.cpu().numpy(), v.cpu().numpy(), cp, ri)
    colcheck.assert_columns(cp, got, ref["mval"], "fp32r")
    colcheck.assert_res2(r2.cpu().numpy(), ref["res2"] + ref["out2"], colcheck.target_column_norms(a0), "fp32r")


@pytest.mark.parametrize("steps", [1, "auto"])
def test_random_numbering(sam, steps):  # noqa: F811
    """Level-3 columns (81 x 49) of a 200^2 mesh whose unknowns are shuffled."""
    mats = [m.to_scipy() for m in W.config2(nx=200, nmat=2, level=1).mats]
    n = mats[0].shape[0]
    p = np.random.default_rng(2).permutation(n)
    mats = [W.CSR.from_scipy(m[p][:, p].tocsr()) for m in mats]
    cp, ri = oracle.pattern(mats[1], 3)
    _check(sam, mats, *_some(cp, ri, n, set(range(0, n, 137))), steps)


@pytest.mark.parametrize("nx,ny", [(90, 90), (91, 90), (128, 64), (129, 64), (128, 128)])
def test_27_point_columns(sam, nx, ny):  # noqa: F811
    """|I| = 125 and 729 entries: the rows of an interior column span
    4 nx ny + 4 nx + 5, from 32,765 to 66,053."""
    mats = [W.CSR.from_scipy(m) for m in _stencil27(nx, ny, 6, nx)]
    cp, ri = oracle.pattern(mats[1], 1)
    _check(sam, mats, *_some(cp, ri, mats[0].n, set(range(0, mats[0].n, 211))), 1)


@pytest.mark.parametrize("m", [23, 30, 32])
def test_columns_over_a_million_rows(sam, m):  # noqa: F811
    """m^2 candidate rows of columns with m unknowns, 1024 (the shadow pass's limit) at most."""
    mats = _spread(1500000, m)
    cp, ri = oracle.pattern(mats[1], 1)
    _check(sam, mats, cp, ri, 1)
