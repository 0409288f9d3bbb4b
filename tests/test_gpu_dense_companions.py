"""A column of the large class (csrc/lsq_dense.cu) gives the same bits whichever
block shape takes it: the shapes that a launch uses depend on the batch."""
import numpy as np
import pytest

from tests.test_gpu_dense_columns import _pair, _window, sam  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("steps", [1, 2, "auto"])
@pytest.mark.parametrize("nj,density", [(40, 0.3), (60, 0.2), (90, 0.3)])
def test_map_alone_and_after_a_sparse_one(sam, nj, density, steps):  # noqa: F811
    """The map alone has a mean |J| above 27 and is solved by small, medium and
    large blocks; after a diagonal map the medium ones are left out."""
    import torch

    n = 175
    mats = _pair(n, density, nj)
    cp, ri = _window(n, nj)
    dcp, dri = _window(n, 1)
    with sam.Handle() as h:
        A0, A1 = (sam.Csr.from_host(m) for m in mats)
        dev = lambda x: torch.from_numpy(np.ascontiguousarray(x)).cuda()  # noqa: E731
        S, D = h.sam_pattern_from_csc(n, dev(cp), dev(ri)), h.sam_pattern_from_csc(n, dev(dcp), dev(dri))
        r1 = torch.empty(n, dtype=torch.float64, device="cuda")
        r2 = torch.empty(2 * n, dtype=torch.float64, device="cuda")
        v1 = h.sam_build(A1, A0, S, "fp32r", steps, res2=r1)[2]
        offs, _, _, v2, _ = h.sam_build_batched([A1, A1], A0, [D, S], "fp32r", steps, res2=r2)
        h.sam_sync()
        assert torch.equal(v1, v2[int(offs[1]):int(offs[2])])
        assert torch.equal(r1, r2[n:])
        S.destroy()
        D.destroy()
