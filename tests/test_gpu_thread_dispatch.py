"""Which builds and adjoints the thread-per-column kernels (csrc/lsq_simt.cu) take:
from 131,072 columns of one structure or 262,144 otherwise, sources of at most
twelve entries per column, whether or not the handle validates them and whether
or not they are symmetric.  The factor tape tells the kernels apart: the Cholesky
factor's diagonal is positive, the QR's is negative where the column's is positive."""
import numpy as np
import pytest
import scipy.sparse as sp

import oracle
from paper_2406_17656_gb300 import workloads as W
from tests import colcheck
from tests.test_gpu_thread_columns import CASES, sam  # noqa: F401

pytestmark = pytest.mark.gpu


def _one_sided(n, k, seed):
    """A diagonal with entries in the k - 1 rows below: unsymmetric, k per column."""
    rng = np.random.default_rng(seed)
    d = [rng.uniform(-1, 0, n - o) if o else np.full(n, k + 1.0) for o in range(k)]
    return sp.diags(d, [-o for o in range(k)]).tocsr()


def _one_long_column(nx, length):
    """A 5-point matrix with one column (and row) of `length` entries."""
    m, c = W.poisson5(nx).to_scipy().tolil(), 5 * nx + 40
    for i in range(length - 5):
        m[3 * nx + 2 * i, c] = m[c, 3 * nx + 2 * i] = -0.01
    m = m.tocsr()
    assert np.diff(m.tocsc().indptr).max() == length
    return W.CSR.from_scipy(m)


LISTS = {
    "width5": CASES["width5"],
    "width9": CASES["width9"],
    "p1": CASES["p1"],
    "width12": CASES["width12"],
    "alone": lambda: (W.config2(nx=513, nmat=1, level=1).mats, 1),                          # 263,169 columns
    "one-sided3": lambda: ([W.CSR.from_scipy(_one_sided(140000, 3, s)) for s in (1, 2)], 1),  # unsymmetric, width 5
    "one-sided5": lambda: ([W.CSR.from_scipy(_one_sided(140000, 5, s)) for s in (1, 2)], 1),
    "long12": lambda: ([_one_long_column(370, 12)] * 2, 1),
    "long13": lambda: ([_one_long_column(370, 13)] * 2, 1),
}


def _call(S, case, trusted):
    import torch

    mats, level = LISTS[case]()
    n, K = mats[0].n, len(mats)
    with S.Handle(trusted=trusted) as h:
        aks = [S.Csr.from_host(m) for m in mats]
        pats = h.sam_pattern_build_batched(aks, level)
        tape = torch.zeros((h.sam_factor_tape_bytes(pats, "fp32r") + 15) // 16 * 4, dtype=torch.float32, device="cuda")
        h.sam_set_factor_tape(S.SAM_TAPE_RECORD, tape)
        r2 = torch.empty(K * n, dtype=torch.float64, device="cuda")
        offs, rp, ci, v, _ = h.sam_build_batched(aks, aks[0], pats, "fp32r", 1, res2=r2)
        h.sam_set_factor_tape(S.SAM_TAPE_OFF)
        g = torch.randn(v.numel(), dtype=torch.float64, device="cuda", generator=torch.Generator("cuda").manual_seed(3))
        da, dz = h.sam_build_backward_batched(aks, [aks[0]] * K, pats, v, g, "fp32r", 1, 0.25)
        h.sam_sync()
        for p in pats:
            p.destroy()
    return mats, level, offs, rp, ci, v, r2, da, dz, tape


@pytest.mark.parametrize("case", list(LISTS))
def test_trusted_and_validating_handles_agree(sam, case):  # noqa: F811
    import torch

    a, b = _call(sam, case, False), _call(sam, case, True)
    for x, y in zip(a[3:9], b[3:9]):
        assert torch.equal(x, y)
    # the first column's first element is R_00: negative from the QR
    for r in (a, b):
        assert (float(r[9][0]) > 0) == (case != "long13")


@pytest.mark.parametrize("trusted", [False, True])
@pytest.mark.parametrize("case", ["one-sided3", "one-sided5", "long12", "long13"])
def test_columns_against_oracle(sam, case, trusted):  # noqa: F811
    mats, level, offs, rp, ci, v, r2, da, dz, _ = _call(sam, case, trusted)
    n = mats[0].n
    k = len(mats) - 1
    part = slice(int(offs[k]), int(offs[k + 1]))
    to_csc = lambda x: colcheck.csr_to_csc_values(n, rp[k * (n + 1):].cpu().numpy(), ci[part].cpu().numpy(),  # noqa: E731
                                                  x[part].cpu().numpy(), cp, ri)
    cp, ri = oracle.pattern(mats[k], level)
    ref = oracle.build(mats[k], mats[0], cp, ri)
    colcheck.assert_columns(cp, to_csc(v), ref["mval"], "fp32r")
    colcheck.assert_res2(r2[k * n:].cpu().numpy(), ref["res2"] + ref["out2"], colcheck.target_column_norms(mats[0]), "fp32r")
    # the adjoint of the oracle's map against the call's (the bar of one step: test_gpu_adjoint.py)
    import torch

    g = torch.randn(v.numel(), dtype=torch.float64, device="cuda", generator=torch.Generator("cuda").manual_seed(3))
    want_k, want_0 = oracle.adjoint(mats[k], mats[0], cp, ri, ref["mval"], to_csc(g), 0.25)
    have_k = da[sum(m.nnz for m in mats[:k]):].cpu().numpy()
    have_0 = dz[k * mats[0].nnz:].cpu().numpy()
    scale = max(np.abs(want_k).max(), np.abs(want_0).max())
    assert np.abs(have_k - want_k).max() <= 1e-7 * scale and np.abs(have_0 - want_0).max() <= 1e-7 * scale


def test_tile_variants_do_not_concern_thread_columns(sam):  # noqa: F811
    """A handle tuned on a small batch (variant 1 of class 1) builds a large one as a
    new handle does; the tuner, run on a large one, leaves its classes at variant 0."""
    import torch

    mats, level = LISTS["width9"]()
    out = []
    for variants in ([0] * 6, [0, 1, 0, 0, 0, 0]):
        with sam.Handle() as h:
            h.sam_set_tile_variants(variants)
            aks = [sam.Csr.from_host(m) for m in mats]
            pats = h.sam_pattern_build_batched(aks, level)
            out.append(h.sam_build_batched(aks, aks[0], pats, "fp32r", 1)[3])
            if variants[1]:
                h.sam_tune(aks, aks[0], pats, "fp32r", 1)
                assert list(h.sam_get_tile_variants())[:2] == [0, 0]
            h.sam_sync()
            for p in pats:
                p.destroy()
    assert torch.equal(*out)
