"""The FP64 column tiles (classes 0-4 of csrc/lsq_core.cuh) at the edges of
their size classes: map, residual, factor tape and adjoint, against the
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


def _mats(n, off, seed):
    rng = np.random.default_rng(seed)
    out = []
    for _ in range(2):
        m = sp.diags([rng.uniform(-1, 1, n - abs(o)) for o in off if o], [o for o in off if o]).tocsr()
        out.append(W.CSR.from_scipy((m + sp.diags(np.asarray(abs(m).sum(1)).ravel() + 1.0)).tocsr()))
    return out


# unknowns per column and half-bandwidth of the source (|I| = nj + 2 b inside)
@pytest.mark.parametrize("nj,b", [(1, 3), (5, 4), (6, 4), (9, 8), (10, 8), (23, 8), (24, 8), (23, 9), (24, 14), (27, 12),
                                  (26, 13), (27, 13), (27, 18), (27, 19)])
def test_class_edges(sam, nj, b):
    import torch

    n = 150
    a0, a1 = _mats(n, sorted({0, 1, -1, b // 2, -(b // 2), b, -b}), 100 * nj + b)
    lo = np.clip(np.arange(n) - nj // 2, 0, n - nj)
    cp = np.arange(n + 1, dtype=np.int32) * nj
    ri = (lo[:, None] + np.arange(nj)[None, :]).astype(np.int32).ravel()
    with sam.Handle() as h:
        Ak, A0 = sam.Csr.from_host(a1), sam.Csr.from_host(a0)
        S = h.sam_pattern_from_csc(n, torch.from_numpy(cp).cuda(), torch.from_numpy(ri).cuda())
        r2 = torch.empty(n, dtype=torch.float64, device="cuda")
        rp, ci, v = h.sam_build(Ak, A0, S, "fp64", 0, res2=r2)
        g = torch.randn(v.numel(), dtype=torch.float64, device="cuda", generator=torch.Generator("cuda").manual_seed(nj))
        dk, d0 = h.sam_build_backward(Ak, A0, S, v, g, "fp64", 0, 0.5)
        tape = torch.zeros(h.sam_factor_tape_bytes([S], "fp64") // 8 + 2, dtype=torch.float64, device="cuda")
        h.sam_set_factor_tape(sam.SAM_TAPE_RECORD, tape)
        v2 = h.sam_build(Ak, A0, S, "fp64", 0)[2]
        h.sam_set_factor_tape(sam.SAM_TAPE_REPLAY, tape)
        dk2, d02 = h.sam_build_backward(Ak, A0, S, v, g, "fp64", 0, 0.5)
        h.sam_set_factor_tape(sam.SAM_TAPE_OFF)
        h.sam_sync()
        S.destroy()
    ref = oracle.build(a1, a0, cp, ri)
    got = colcheck.csr_to_csc_values(n, rp.cpu().numpy(), ci.cpu().numpy(), v.cpu().numpy(), cp, ri)
    colcheck.assert_columns(cp, got, ref["mval"], "fp64")
    colcheck.assert_res2(r2.cpu().numpy(), ref["res2"] + ref["out2"], colcheck.target_column_norms(a0), "fp64")
    assert torch.equal(v, v2) and torch.equal(dk, dk2) and torch.equal(d0, d02)
    # <g, dM> along a direction of (A_k, A_0), by central differences of the
    # oracle's map: truncation h^2 and rounding u / h, 1e-10 at h = 1e-5, times
    # the third derivative of a map whose diagonal dominance is above 1
    rng = np.random.default_rng(7)
    uk, u0 = rng.standard_normal(a1.nnz), rng.standard_normal(a0.nnz)
    gm = colcheck.csr_to_csc_values(n, rp.cpu().numpy(), ci.cpu().numpy(), g.cpu().numpy(), cp, ri)
    step = 1e-5

    def loss(s):
        k = W.CSR(n, a1.indptr, a1.indices, a1.data + s * step * uk)
        z = W.CSR(n, a0.indptr, a0.indices, a0.data + s * step * u0)
        r = oracle.build(k, z, cp, ri)
        return float(gm @ r["mval"]) + 0.5 * float((r["res2"] + r["out2"]).sum())

    want = (loss(1) - loss(-1)) / (2 * step)
    have = float(dk.cpu().numpy() @ uk + d0.cpu().numpy() @ u0)
    scale = np.linalg.norm(dk.cpu().numpy()) * np.linalg.norm(uk) + np.linalg.norm(d0.cpu().numpy()) * np.linalg.norm(u0)
    assert abs(have - want) <= 1e-7 * scale
