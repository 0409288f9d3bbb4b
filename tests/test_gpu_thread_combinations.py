"""The thread-per-column kernels and the large class in the calls that reach them
with paths of their own: captured plans (copies rewritten at every replay), host
outputs in chunks of maps (work list by map, lists cleared per chunk), and columns
of nine unknowns with eleven entries each (the widest copies)."""
import numpy as np
import pytest

import oracle
from paper_2406_17656_gb300 import workloads as W
from tests import colcheck
from tests.test_gpu_thread_columns import _band11
from tests.test_gpu_thread_dispatch import LISTS, sam  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("case,trusted,steps", [("width9", False, 1), ("width9", True, 2), ("width5", False, "auto"),
                                                ("p1", False, 1), ("p1", True, "auto"), ("one-sided5", False, 1),
                                                ("long13", True, 1)])
def test_plan_replays_equal_direct_builds(sam, case, trusted, steps):  # noqa: F811
    import torch

    mats, level = LISTS[case]()
    n, K = mats[0].n, len(mats)
    with sam.Handle(trusted=trusted) as h:
        aks = [sam.Csr.from_host(m) for m in mats]
        pats = h.sam_pattern_build_batched(aks, level)
        plan = h.sam_plan_create(aks, aks[0], pats, "fp32r", steps, want_status=True, want_res2=True)
        for factor in (1.0, 1.25):
            for a in aks[1:]:
                a.data.mul_(factor)
            plan.execute()
            st = torch.empty(K * n, dtype=torch.int32, device="cuda")
            r2 = torch.empty(K * n, dtype=torch.float64, device="cuda")
            _, rp, ci, v, _ = h.sam_build_batched(aks, aks[0], pats, "fp32r", steps, col_status=st, res2=r2)
            h.sam_sync()
            assert torch.equal(plan.M_row_ptr, rp) and torch.equal(plan.M_col_idx, ci) and torch.equal(plan.M_val, v)
            assert torch.equal(plan.col_status, st) and torch.equal(plan.res2, r2) and not bool(st.any())
        plan.destroy()
        for p in pats:
            p.destroy()


@pytest.mark.parametrize("nx,nmat,level,steps", [(182, 8, 1, 1), (182, 9, 1, 2), (182, 8, 1, "auto"), (256, 5, 3, 1)])
@pytest.mark.parametrize("trusted", [False, True])
def test_chunked_host_outputs_equal_device_outputs(sam, nx, nmat, level, steps, trusted):  # noqa: F811
    import torch

    mats = W.config2(nx=nx, nmat=nmat, level=level).mats
    n = mats[0].n
    assert n * nmat >= 2 << 17
    with sam.Handle(trusted=trusted) as h:
        aks = [sam.Csr.from_host(m) for m in mats]
        pats = h.sam_pattern_build_batched(aks, level)
        r2 = torch.empty(nmat * n, dtype=torch.float64, device="cuda")
        offs, rp, ci, v, fro = h.sam_build_batched(aks, aks[0], pats, "fp32r", steps, res2=r2, want_fro=True)
        out = [torch.empty(x.shape, dtype=x.dtype).pin_memory() for x in (rp, ci, v, r2)]
        fro_h = h.sam_build_batched(aks, aks[0], pats, "fp32r", steps, M_row_ptr=out[0], M_col_idx=out[1], M_val=out[2],
                                    res2=out[3], want_fro=True, offsets=offs)[4]
        for p in pats:
            p.destroy()
    for got, want in zip(out, (rp, ci, v, r2)):
        assert torch.equal(got, want.cpu())
    assert np.array_equal(fro, fro_h)


@pytest.mark.parametrize("steps", [1, 2])
def test_nine_unknowns_of_eleven_entries(sam, steps):  # noqa: F811
    """|I| = 19 and 99 entries in interior columns: map and adjoint against the
    oracle, the bars of test_gpu_adjoint.py."""
    import torch

    n, nj, rho = 140000, 9, 0.5
    mats = _band11(n, 1) + [W.CSR(n, *(lambda m: (m.indptr, m.indices, m.data * (1 + 0.1 * np.cos(np.arange(m.nnz)))))(
        _band11(n, 1)[0]))]
    lo = np.clip(np.arange(n) - nj // 2, 0, n - nj)
    cp = np.arange(n + 1, dtype=np.int32) * nj
    ri = (lo[:, None] + np.arange(nj)[None, :]).astype(np.int32).ravel()
    with sam.Handle() as h:
        aks = [sam.Csr.from_host(m) for m in mats]
        S = h.sam_pattern_from_csc(n, torch.from_numpy(cp).cuda(), torch.from_numpy(ri).cuda())
        r2 = torch.empty(2 * n, dtype=torch.float64, device="cuda")
        offs, rp, ci, v, _ = h.sam_build_batched(aks, aks[0], [S, S], "fp32r", steps, res2=r2)
        g = torch.randn(v.numel(), dtype=torch.float64, device="cuda", generator=torch.Generator("cuda").manual_seed(5))
        da, dz = h.sam_build_backward_batched(aks, [aks[0]] * 2, [S, S], v, g, "fp32r", steps, rho)
        h.sam_sync()
        S.destroy()
    part = slice(int(offs[1]), int(offs[2]))
    to_csc = lambda x: colcheck.csr_to_csc_values(n, rp[n + 1:].cpu().numpy(), ci[part].cpu().numpy(),  # noqa: E731
                                                  x[part].cpu().numpy(), cp, ri)
    ref = oracle.build(mats[1], mats[0], cp, ri)
    colcheck.assert_columns(cp, to_csc(v), ref["mval"], "fp32r")
    colcheck.assert_res2(r2[n:].cpu().numpy(), ref["res2"] + ref["out2"], colcheck.target_column_norms(mats[0]), "fp32r")
    want_k, want_0 = oracle.adjoint(mats[1], mats[0], cp, ri, ref["mval"], to_csc(g), rho)
    nz = mats[0].nnz
    scale = max(np.abs(want_k).max(), np.abs(want_0).max())
    tol = 1e-7 if steps == 1 else 1e-10
    assert np.abs(da[nz:].cpu().numpy() - want_k).max() <= tol * scale
    assert np.abs(dz[nz:].cpu().numpy() - want_0).max() <= tol * scale
