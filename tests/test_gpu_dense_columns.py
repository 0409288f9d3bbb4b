"""The large class of refined FP32 builds (csrc/lsq_dense.cu) at the edges of
its three block shapes: 52 / 53 unknowns, 127 / 128, values that do not fit
beside the lists, rows that span most of a large matrix, and columns that
break down, against the oracle column by column."""
import numpy as np
import pytest
import scipy.sparse as sp

import oracle
from paper_2406_17656_gb300 import workloads as W
from tests import colcheck

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def sam():
    torch = pytest.importorskip("torch")
    from paper_2406_17656_gb300 import build, sam as S

    build.build()
    assert torch.cuda.is_available()
    return S


def _pair(n, density, seed):
    rng = np.random.default_rng(seed)
    p = rng.random((n, n)) < density
    np.fill_diagonal(p, True)
    out = []
    for _ in range(2):
        a = np.where(p, rng.uniform(-1, 1, (n, n)), 0.0)
        np.fill_diagonal(a, np.abs(a).sum(1) + 1.0)
        i, j = np.nonzero(p)
        out.append(W.CSR.from_scipy(sp.csr_matrix((a[i, j], (i, j)), shape=(n, n))))
    return out


def _window(n, nj):
    """A pattern of nj consecutive rows around the diagonal in every column."""
    lo = np.clip(np.arange(n) - nj // 2, 0, n - nj)
    cp = np.arange(n + 1, dtype=np.int32) * nj
    return cp, (lo[:, None] + np.arange(nj)[None, :]).astype(np.int32).ravel()


def _spread(n=300000, m=30):
    """A diagonal with m random rows and columns coupled densely (m^2 = 900
    candidate rows: the shadow pass takes 1024 past a span of 32768): their column
    problems' rows span the whole matrix."""
    rng = np.random.default_rng(4)
    s = np.sort(rng.choice(n, m, replace=False))
    out = []
    for _ in range(2):
        i, j = np.meshgrid(s, s, indexing="ij")
        off = sp.csr_matrix((rng.uniform(-1, 1, m * m), (i.ravel(), j.ravel())), shape=(n, n))
        out.append(W.CSR.from_scipy(off + sp.diags(np.full(n, 2.0 * m))))
    return out


def _check(sam, mats, cp, ri, steps, cols=None):
    import torch

    a1, a0 = mats[1], mats[0]
    n = a0.n
    with sam.Handle() as h:
        Ak, A0 = sam.Csr.from_host(a1), sam.Csr.from_host(a0)
        S = h.sam_pattern_from_csc(n, torch.from_numpy(cp).cuda(), torch.from_numpy(ri).cuda())
        r2 = torch.empty(n, dtype=torch.float64, device="cuda")
        rp, ci, v = h.sam_build(Ak, A0, S, "fp32r", steps, res2=r2)
        h.sam_sync()
        S.destroy()
    ref = oracle.build(a1, a0, cp, ri)
    got = colcheck.csr_to_csc_values(n, rp.cpu().numpy(), ci.cpu().numpy(), v.cpu().numpy(), cp, ri)
    colcheck.assert_columns(cp, got, ref["mval"], "fp32r", cols=cols)
    colcheck.assert_res2(r2.cpu().numpy(), ref["res2"] + ref["out2"], colcheck.target_column_norms(a0), "fp32r")


@pytest.mark.parametrize("steps", [1, 2, "auto"])
@pytest.mark.parametrize("n,nj,density", [(170, 52, 0.04), (170, 53, 0.04), (150, 28, 0.2), (160, 127, 0.1),
                                          (160, 128, 0.1), (175, 90, 1.0)])
def test_windows(sam, n, nj, density, steps):
    mats = _pair(n, density, 10 * n + nj)
    cp, ri = _window(n, nj)
    _check(sam, mats, cp, ri, steps)


def test_rows_far_apart(sam):
    mats = _spread()
    cp, ri = oracle.pattern(mats[1], 1)
    _check(sam, mats, cp, ri, 1)


@pytest.mark.parametrize("nj", [40, 60])
def test_breakdown_and_zero_columns(sam, nj):
    """Two nearly equal columns (kappa about 1e9: no FP32 factor) are solved in
    FP64; a zero column is rank deficient where it is an unknown."""
    import torch

    mats = _pair(170, 0.2, 77)
    m = mats[1].to_scipy().tocsc()
    d = m.toarray()
    d[:, 31] = d[:, 30] * (1.0 + 1e-9 * np.random.default_rng(1).uniform(-1, 1, 170))
    d[:, 120] = 0.0
    i, j = np.nonzero((mats[1].dense() != 0) | (d != 0))
    a1 = W.CSR.from_scipy(sp.csr_matrix((d[i, j], (i, j)), shape=(170, 170)))
    cp, ri = _window(170, nj)
    with sam.Handle() as h:
        S = h.sam_pattern_from_csc(170, torch.from_numpy(cp).cuda(), torch.from_numpy(ri).cuda())
        st = torch.empty(170, dtype=torch.int32, device="cuda")
        h.sam_build(sam.Csr.from_host(a1), sam.Csr.from_host(mats[0]), S, "fp32r", 1, col_status=st)
        with pytest.raises(sam.SamError):
            h.sam_sync()
        solved64 = h.sam_refine_stats()[2]
        S.destroy()
    rows = ri.reshape(170, nj)
    st = st.cpu().numpy()
    assert np.array_equal(st == sam.SAM_ERR_RANK_DEFICIENT, (rows == 120).any(1))
    both = (rows == 30).any(1) & (rows == 31).any(1) & ~(rows == 120).any(1)
    assert both.any() and not st[both].any() and solved64 >= both.sum()
