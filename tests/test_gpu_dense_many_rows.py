"""Large-class columns (csrc/lsq_dense.cu) of few unknowns and some 200 to 500 rows:
against the oracle, and alone (more than 256 entries in the mean B: medium blocks)
as after a diagonal map (none), bit for bit."""
import numpy as np
import pytest

from tests.test_gpu_dense_columns import _check, _pair, _window, sam  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nj,density", [(2, 0.25), (5, 0.2), (14, 0.1)])
def test_few_unknowns_and_many_rows(sam, nj, density):  # noqa: F811
    import torch

    n = 600
    mats = _pair(n, density, nj)
    cp, ri = _window(n, nj)
    _check(sam, mats, cp, ri, 1)
    dcp, dri = _window(n, 1)
    dev = lambda x: torch.from_numpy(np.ascontiguousarray(x)).cuda()  # noqa: E731
    with sam.Handle() as h:
        A0, A1 = (sam.Csr.from_host(m) for m in mats)
        S, D = h.sam_pattern_from_csc(n, dev(cp), dev(ri)), h.sam_pattern_from_csc(n, dev(dcp), dev(dri))
        r1 = torch.empty(n, dtype=torch.float64, device="cuda")
        r2 = torch.empty(2 * n, dtype=torch.float64, device="cuda")
        v1 = h.sam_build(A1, A0, S, "fp32r", 1, res2=r1)[2]
        offs, _, _, v2, _ = h.sam_build_batched([A1, A1], A0, [D, S], "fp32r", 1, res2=r2)
        h.sam_sync()
        assert torch.equal(v1, v2[int(offs[1]):int(offs[2])]) and torch.equal(r1, r2[n:])
        S.destroy()
        D.destroy()
