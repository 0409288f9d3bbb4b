"""The thread-per-column adjoint (csrc/lsq_simt.cu) where its Cholesky factor
contracts slowly: coefficients with contrast and rows scaled by up to 10 (extra
corrections), up to 1000 (some or nearly all columns are left to the QR tiles), one
unscaled map beside them, and columns that are rank deficient, against the oracle's
adjoint and the single maps' calls."""
import numpy as np
import pytest
import scipy.sparse as sp

import oracle
from paper_2406_17656_gb300 import workloads as W
from tests.test_gpu_thread_columns import sam  # noqa: F401

pytestmark = pytest.mark.gpu


def _scaled(mats, a):
    out = [mats[0]]
    for k, m in enumerate(mats[1:]):
        s = 10.0 ** np.random.default_rng(50 + k).uniform(-a, a, m.n)
        out.append(W.CSR.from_scipy(sp.diags(s) @ m.to_scipy()))
    return out


def _contrast(nx, K):
    """5-point diffusion with a coefficient of exp(N(0, 1.5^2)) per node."""
    out = []
    for k in range(K):
        c = np.exp(1.5 * np.random.default_rng(k).standard_normal(nx * nx))
        m = W.poisson5(nx).to_scipy().tocoo()
        off = m.row != m.col
        v = -0.5 * (c[m.row[off]] + c[m.col[off]])
        L = sp.coo_matrix((v, (m.row[off], m.col[off])), shape=m.shape).tocsr()
        out.append(W.CSR.from_scipy((L + sp.diags(c - np.asarray(L.sum(1)).ravel())).tocsr()))
    return out


CASES = {
    "contrast": (lambda: _contrast(182, 4), True),
    "rows0.5": (lambda: _scaled(W.config2(nx=182, nmat=4, level=1).mats, 0.5), True),
    "rows1": (lambda: _scaled(W.config2(nx=182, nmat=4, level=1).mats, 1.0), False),
    "rows2": (lambda: _scaled(W.config2(nx=182, nmat=4, level=1).mats, 2.0), False),
    "rows3": (lambda: _scaled(W.config2(nx=182, nmat=4, level=1).mats, 3.0), False),
}


@pytest.mark.parametrize("steps", [1, 2])
@pytest.mark.parametrize("case", list(CASES))
def test_against_the_oracle_and_single_calls(sam, case, steps):  # noqa: F811
    """The bars of test_gpu_adjoint.py where every column's rho allows them; where
    it does not, the batch is no further from the oracle than twice the single
    calls (the QR tiles) and the bar."""
    import torch

    make, bar = CASES[case]
    mats = make()
    n, K, rho = mats[0].n, len(mats), 0.5
    assert n < 1 << 17 <= n * K
    rng = np.random.default_rng(7)
    p = oracle.pattern(mats[0], 1)
    fwd = [oracle.build(m, mats[0], *p)["mval"] for m in mats]
    gbar = [rng.standard_normal(len(p[1])) for _ in mats]
    to_csr = lambda x: torch.from_numpy(oracle.to_csr(n, p[0], p[1], x)[2]).cuda()  # noqa: E731
    ms, gs = [to_csr(x) for x in fwd], [to_csr(x) for x in gbar]
    tol = 1e-7 if steps == 1 else 1e-10
    with sam.Handle() as h:
        aks = [sam.Csr.from_host(m) for m in mats]
        pats = h.sam_pattern_build_batched(aks, 1)
        da, dz = h.sam_build_backward_batched(aks, [aks[0]] * K, pats, torch.cat(ms), torch.cat(gs), "fp32r", steps, rho)
        h.sam_sync()
        nz = aks[0].nnz
        for k in range(K):
            dk1, d01 = h.sam_build_backward(aks[k], aks[0], pats[k], ms[k], gs[k], "fp32r", steps, rho)
            h.sam_sync()
            want_k, want_0 = oracle.adjoint(mats[k], mats[0], *p, fwd[k], gbar[k], rho)
            scale = max(np.abs(want_k).max(), np.abs(want_0).max())
            for got, one, want in ((da[k * nz:(k + 1) * nz], dk1, want_k), (dz[k * nz:(k + 1) * nz], d01, want_0)):
                err = np.abs(got.cpu().numpy() - want).max() / scale
                qr = np.abs(one.cpu().numpy() - want).max() / scale
                assert err <= (tol if bar else 2 * qr + tol)


def test_rank_deficient_columns(sam):  # noqa: F811
    """A column of zeros in one map: its columns report it as the single call does,
    and every other column's gradient is the same."""
    import torch

    mats = W.config2(nx=182, nmat=4, level=1).mats
    n, K = mats[0].n, len(mats)
    data = mats[2].data.copy()
    data[mats[2].indices == 5000] = 0.0
    mats = mats[:2] + [W.CSR(n, mats[2].indptr, mats[2].indices, data)] + mats[3:]
    with sam.Handle() as h:
        aks = [sam.Csr.from_host(m) for m in mats]
        pats = h.sam_pattern_build_batched(aks, 1)
        v = h.sam_build_batched(aks, aks[0], pats, "fp32r", 2)[3]
        with pytest.raises(sam.SamError):
            h.sam_sync()
        g = torch.randn(v.numel(), dtype=torch.float64, device="cuda", generator=torch.Generator("cuda").manual_seed(1))
        da, dz = h.sam_build_backward_batched(aks, [aks[0]] * K, pats, v, g, "fp32r", 2, 0.5)
        with pytest.raises(sam.SamError):
            h.sam_sync()
        e, nz = v.numel() // K, aks[0].nnz
        for k in range(K):
            one = h.sam_build_backward(aks[k], aks[0], pats[k], v[k * e:(k + 1) * e], g[k * e:(k + 1) * e], "fp32r", 2, 0.5)
            if k == 2:
                with pytest.raises(sam.SamError):
                    h.sam_sync()
            else:
                h.sam_sync()
            scale = max(float(x.abs().max()) for x in one)
            assert float((da[k * nz:(k + 1) * nz] - one[0]).abs().max()) <= 1e-10 * scale
            assert float((dz[k * nz:(k + 1) * nz] - one[1]).abs().max()) <= 1e-10 * scale
