"""Builds and adjoints that nearly fill the device: the copies of the
thread-per-column kernels (csrc/lsq_simt.cu) are optional, so a batch that takes
them runs wherever one that does not (one column of 13 entries, otherwise the same)
runs, on the register tiles if there is no room."""
import numpy as np
import pytest

from paper_2406_17656_gb300 import workloads as W
from tests.test_gpu_thread_dispatch import _one_long_column, sam  # noqa: F401

pytestmark = pytest.mark.gpu
K, NX, STEP = 4, 512, 4 << 20


def _calls(S, kind, trusted):
    """Inputs and outputs on the device; returns run(), which makes the call on a
    new handle and returns its map or gradient values."""
    import torch

    out = {}
    for name, m in (("short", W.poisson5(NX)), ("long", _one_long_column(NX, 13))):
        mats = [W.CSR(m.n, m.indptr, m.indices, m.data * (1.0 + 0.1 * k)) for k in range(K)]
        with S.Handle() as h:
            aks = [S.Csr.from_host(x) for x in mats]
            p = h.sam_pattern_build(aks[0], 1)
            cp, ri = torch.as_tensor(p.colptr(), device="cuda").clone(), torch.as_tensor(p.rowidx(), device="cuda").clone()
            nnz = p.nnz
            v0 = h.sam_build_batched(aks, aks[0], [p] * K, "fp32r", 1)[3]
            h.sam_sync()
            p.destroy()
        n = mats[0].n
        rp = torch.empty(K * (n + 1), dtype=torch.int32, device="cuda")
        ci = torch.empty(K * nnz, dtype=torch.int32, device="cuda")
        v = torch.empty(K * nnz, dtype=torch.float64, device="cuda")
        da, dz = (torch.empty(K * mats[0].nnz, dtype=torch.float64, device="cuda") for _ in range(2))
        offs = np.arange(K + 1, dtype=np.int64) * nnz

        def run(aks=aks, cp=cp, ri=ri, v0=v0, rp=rp, ci=ci, v=v, da=da, dz=dz, offs=offs, n=n):
            h = S.Handle(trusted=trusted)
            try:
                p = h.sam_pattern_from_csc(n, cp, ri)
                try:
                    if kind == "build":
                        h.sam_build_batched(aks, aks[0], [p] * K, "fp32r", 1, M_row_ptr=rp, M_col_idx=ci, M_val=v, offsets=offs)
                        res = v
                    elif kind == "adjoint":
                        h.sam_build_backward_batched(aks, [aks[0]] * K, [p] * K, v0, v0, "fp32r", 1, 0.5, dA_k_val=da, dA_0_val=dz)
                        res = da
                    h.sam_sync()
                finally:
                    p.destroy()
                return res
            finally:
                h.close()

        out[name] = run
    return out


@pytest.mark.parametrize("kind", ["build", "adjoint"])
def test_runs_wherever_the_register_tiles_run(sam, kind):  # noqa: F811
    import torch

    runs = _calls(sam, kind, False)
    want = {k: f().clone() for k, f in runs.items()}  # (and every kernel is loaded)
    torch.cuda.synchronize()
    torch.cuda.empty_cache()

    def attempt(name, room):
        """The call with `room` bytes of the device free: its values, or None."""
        free = torch.cuda.mem_get_info()[0]
        fill = torch.empty(max(free - room, 1), dtype=torch.uint8, device="cuda")
        try:
            return runs[name]()
        except sam.SamError as e:
            assert e.status == sam.SAM_ERR_OOM
            return None
        finally:
            del fill
            torch.cuda.empty_cache()

    lo, hi = 0, 4 << 30
    assert attempt("long", hi) is not None
    while hi - lo > STEP:
        mid = (lo + hi) // 2
        if attempt("long", mid) is None:
            lo = mid
        else:
            hi = mid
    tiles = 0
    for room in (hi + STEP, hi + 8 * STEP, hi + 24 * STEP, hi + 64 * STEP):
        got = attempt("short", room)
        assert got is not None, "no room at %d bytes, %d suffice without the copies" % (room, hi)
        err = float((got - want["short"]).norm() / want["short"].norm())
        assert err <= (1e-10 if kind == "build" else 1e-7)
        tiles += not torch.equal(got, want["short"])
    assert 1 <= tiles <= 3  # the register tiles at the limit, the copies where there is room
