"""The thread-per-column kernels of refined FP32 builds and their adjoint
(csrc/lsq_simt.cu), which take the two smallest size classes of batches of
32,768 columns or more: every width of its value copy, orders that are no multiple of 32, one
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
    "width5": lambda: (_poisson(182, 4), 1),                       # 4 x 33124
    "width7": lambda: (W.config3(nx=33, nmat=4).mats, 1),          # 4 x 35937
    "width9": lambda: (W.config2(nx=182, nmat=4, level=1).mats, 1),  # 4 x 33124
    "width12": lambda: (_band11(262201, 1), 0),                     # one map, one unknown per column
    "p1": lambda: (W.config4(ncell=300, nmat=3).mats, 1),          # separate structures
    "scaled": lambda: (_scaled(W.config2(nx=182, nmat=4, level=1).mats), 1),
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
    assert n * K >= 1 << 17
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

    mats = W.config2(nx=182, nmat=4, level=1).mats
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


@pytest.mark.parametrize("steps", [1, 2])
@pytest.mark.parametrize("case", ["width5", "width7", "width9", "p1", "scaled"])
def test_adjoint(sam, case, steps):
    """The batched adjoint against the oracle's (the bars of test_gpu_adjoint.py)
    and against the single maps' calls, which are below the batch size (the QR
    kernel).  The rows of "scaled" make every column of the scaled maps one that
    the thread-per-column kernel leaves: there only the calls are compared, and
    both solve those columns alike."""
    import torch

    mats, level = CASES[case]()
    n, K = mats[0].n, len(mats)
    assert n < 1 << 17 <= n * K
    rho = 0.5
    rng = np.random.default_rng(7)
    pat = [oracle.pattern(m, level) for m in mats]
    fwd = [oracle.build(m, mats[0], *p)["mval"] for m, p in zip(mats, pat)]
    gbar = [rng.standard_normal(len(p[1])) for p in pat]
    to_csr = lambda p, x: torch.from_numpy(oracle.to_csr(n, p[0], p[1], x)[2]).cuda()  # noqa: E731
    ms = [to_csr(p, x) for p, x in zip(pat, fwd)]
    gs = [to_csr(p, x) for p, x in zip(pat, gbar)]
    tol = 1e-7 if steps == 1 else 1e-10
    with sam.Handle() as h:
        aks = [sam.Csr.from_host(m) for m in mats]
        pats = h.sam_pattern_build_batched(aks, level)
        dmr = torch.empty(sum(m.numel() for m in ms), dtype=torch.float64, device="cuda")
        da, dz = h.sam_build_backward_batched(aks, [aks[0]] * K, pats, torch.cat(ms), torch.cat(gs), "fp32r", steps, rho,
                                              dM_resid=dmr)
        h.sam_sync()
        ea = em = 0
        nz = aks[0].nnz
        for k in range(K):
            dk, d0 = da[ea:ea + aks[k].nnz], dz[k * nz:(k + 1) * nz]
            one = torch.empty_like(ms[k])
            dk1, d01 = h.sam_build_backward(aks[k], aks[0], pats[k], ms[k], gs[k], "fp32r", steps, rho, dM_resid=one)
            h.sam_sync()
            scale = max(float(dk1.abs().max()), float(d01.abs().max()))
            assert float((dk - dk1).abs().max()) <= tol * scale and float((d0 - d01).abs().max()) <= tol * scale
            assert float((dmr[em:em + one.numel()] - one).abs().max()) <= 1e-9 * max(1.0, float(one.abs().max()))
            if case != "scaled":
                want_k, want_0 = oracle.adjoint(mats[k], mats[0], *pat[k], fwd[k], gbar[k], rho)
                scale = max(np.abs(want_k).max(), np.abs(want_0).max())
                assert np.abs(dk.cpu().numpy() - want_k).max() <= tol * scale
                assert np.abs(d0.cpu().numpy() - want_0).max() <= tol * scale
            ea += aks[k].nnz
            em += one.numel()


def test_factor_tape_of_a_large_batch(sam):
    """Recording changes nothing in the build, the recorded R of every column
    is a factor of its B^T B, and a replaying adjoint equals the recomputing one."""
    import torch

    mats = W.config2(nx=182, nmat=4, level=1).mats
    n, K = mats[0].n, len(mats)
    with sam.Handle() as h:
        aks = [sam.Csr.from_host(m) for m in mats]
        pats = h.sam_pattern_build_batched(aks, 1)
        _, _, _, v, _ = h.sam_build_batched(aks, aks[0], pats, "fp32r", 1)
        tape = torch.zeros((h.sam_factor_tape_bytes(pats, "fp32r") + 15) // 16 * 4, dtype=torch.float32, device="cuda")
        h.sam_set_factor_tape(sam.SAM_TAPE_RECORD, tape)
        _, _, _, v2, _ = h.sam_build_batched(aks, aks[0], pats, "fp32r", 1)
        h.sam_set_factor_tape(sam.SAM_TAPE_REPLAY, tape)
        g = torch.randn(v.numel(), dtype=torch.float64, device="cuda", generator=torch.Generator("cuda").manual_seed(3))
        r1 = h.sam_build_backward_batched(aks, [aks[0]] * K, pats, v, g, "fp32r", 1, 0.25)
        h.sam_set_factor_tape(sam.SAM_TAPE_OFF)
        r2 = h.sam_build_backward_batched(aks, [aks[0]] * K, pats, v, g, "fp32r", 1, 0.25)
        h.sam_sync()
        assert torch.equal(v, v2) and torch.equal(r1[0], r2[0]) and torch.equal(r1[1], r2[1])
    cp, ri = oracle.pattern(mats[0], 1)
    nj = np.diff(cp)
    slot = np.concatenate([[0], np.cumsum((nj * (nj + 1) // 2 + 3) & ~3)])
    t = tape.cpu().numpy().astype(np.float64)
    a = mats[3].to_scipy().tocsc()
    for j in np.random.default_rng(1).integers(0, n, 200):
        B = a[:, ri[cp[j]:cp[j + 1]]].toarray()
        B = B[np.any(B != 0, axis=1)]
        m = nj[j]
        R = np.zeros((m, m))
        R[np.triu_indices(m)] = t[3 * slot[-1] + slot[j]:][:m * (m + 1) // 2]
        G = B.T @ B
        assert np.abs(R.T @ R - G).max() <= 30 * m * 2.0**-24 * np.abs(G).max()
