"""The thread-per-column kernel of refined FP32 builds (csrc/lsq_simt.cu),
which takes the two smallest size classes of batches of 32,768 columns or
more: every width of its value copy, orders that are no multiple of 32, one
shared structure and separate ones, and columns that break down, against the
oracle column by column."""
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


def _band11(n, nmat):
    """Eleven entries per interior column, structurally symmetric."""
    rng = np.random.default_rng(3)
    mats = []
    for _ in range(nmat):
        d = [rng.uniform(-1, 1, n - abs(o)) if o else np.full(n, 12.0) for o in range(-5, 6)]
        mats.append(W.CSR.from_scipy(sp.diags(d, range(-5, 6)).tocsr()))
    return mats


def _scaled(mats):
    """Row scales over 1e-3..1e3 on every matrix but the first (condition
    numbers up to 1e6: the FP32 factor breaks down or the guard sends the
    column to the FP64 re-solve)."""
    out = [mats[0]]
    for k, m in enumerate(mats[1:]):
        s = 10.0 ** np.random.default_rng(50 + k).uniform(-3, 3, m.n)
        out.append(W.CSR.from_scipy(sp.diags(s) @ m.to_scipy()))
    return out


CASES = {
    "width5": lambda: (_poisson(101, 4), 1),                       # 4 x 10201
    "width7": lambda: (W.config3(nx=21, nmat=4).mats, 1),          # 4 x 9261
    "width9": lambda: (W.config2(nx=97, nmat=4, level=1).mats, 1),  # 4 x 9409
    "width12": lambda: (_band11(33001, 1), 0),                     # one map, one unknown per column
    "p1": lambda: (W.config4(ncell=105, nmat=3).mats, 1),          # separate structures
    "scaled": lambda: (_scaled(W.config2(nx=97, nmat=4, level=1).mats), 1),
}


def _poisson(nx, nmat):
    a0 = W.poisson5(nx)
    d = np.random.default_rng(8)
    return [a0] + [W.CSR.from_scipy(a0.to_scipy() + sp.diags(d.uniform(0, 0.5, a0.n))) for _ in range(nmat - 1)]


@pytest.mark.parametrize("steps", [1, 2, "auto"])
@pytest.mark.parametrize("case", list(CASES))
def test_columns_against_oracle(sam, case, steps):
    import torch

    mats, level = CASES[case]()
    n, K = mats[0].n, len(mats)
    assert n * K >= 32768
    with sam.Handle() as h:
        aks = [sam.Csr.from_host(m) for m in mats]
        pats = h.sam_pattern_build_batched(aks, level)
        st = torch.empty(K * n, dtype=torch.int32, device="cuda")
        r2 = torch.empty(K * n, dtype=torch.float64, device="cuda")
        offs, rp, ci, v, _ = h.sam_build_batched(aks, aks[0], pats, "fp32r", steps, col_status=st, res2=r2)
        h.sam_sync()
        rp, ci, v, r2 = rp.cpu().numpy(), ci.cpu().numpy(), v.cpu().numpy(), r2.cpu().numpy()
        assert int(st.abs().max()) == 0
        gamma = colcheck.target_column_norms(mats[0])
        for k, m in enumerate(mats):
            cp, ri = oracle.pattern(m, level)
            ref = oracle.build(m, mats[0], cp, ri)
            got = colcheck.csr_to_csc_values(n, rp[k * (n + 1):(k + 1) * (n + 1)], ci[offs[k]:offs[k + 1]],
                                             v[offs[k]:offs[k + 1]], cp, ri)
            colcheck.assert_columns(cp, got, ref["mval"], "fp32r", what="map %d" % k)
            colcheck.assert_res2(r2[k * n:(k + 1) * n], ref["res2"] + ref["out2"], gamma, "fp32r")


def test_zero_and_nonfinite_columns(sam):
    """A column of zeros is rank deficient and a NaN is non-finite in every
    column problem that holds it; all others are solved."""
    import torch

    mats = W.config2(nx=97, nmat=4, level=1).mats
    n, K = mats[0].n, len(mats)
    data = mats[2].data.copy()
    data[mats[2].indices == 5000] = 0.0
    data[(mats[2].indices == 7000) & (np.repeat(np.arange(n), np.diff(mats[2].indptr)) == 7000)] = np.nan
    mats = mats[:2] + [W.CSR(n, mats[2].indptr, mats[2].indices, data)] + mats[3:]
    with sam.Handle() as h:
        aks = [sam.Csr.from_host(m) for m in mats]
        pats = h.sam_pattern_build_batched(aks, 1)
        st = torch.empty(K * n, dtype=torch.int32, device="cuda")
        h.sam_build_batched(aks, aks[0], pats, "fp32r", 1, col_status=st)
        with pytest.raises(sam.SamError):
            h.sam_sync()
    s = st.cpu().numpy().reshape(K, n)
    cp, ri = oracle.pattern(mats[0], 1)
    holds = lambda c: {j for j in range(n) if c in ri[cp[j]:cp[j + 1]]}  # noqa: E731
    assert set(np.flatnonzero(s[2] == sam.SAM_ERR_RANK_DEFICIENT)) == holds(5000)
    assert set(np.flatnonzero(s[2] == sam.SAM_ERR_NONFINITE)) == holds(7000)
    assert not s[[0, 1, 3]].any()
