"""The large class of refined FP32 builds (csrc/lsq_dense.cu) on matrices whose
entries are far from 1: down to where B^T B leaves FP32's range (1e-19) and the
columns are solved in FP64, against the oracle column by column."""
import numpy as np
import pytest

from paper_2406_17656_gb300 import workloads as W
from tests.test_gpu_dense_columns import _check, _pair, _window, sam  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("steps", [1, "auto"])
@pytest.mark.parametrize("scale_k,scale_0", [(1e-15, 1e-15), (1e-18, 1e-18), (1e-18, 1.0), (1e-19, 1e-19), (3e-20, 3e-20),
                                             (1e-21, 1.0), (1e-23, 1e-23), (1e-25, 1.0), (1e-25, 1e-25), (1e12, 1e-12),
                                             (1e15, 1e15), (1.0, 1e-30)])
def test_scaled_matrices(sam, scale_k, scale_0, steps):  # noqa: F811
    a0, a1 = _pair(170, 0.2, 3)
    mats = [W.CSR(170, a0.indptr, a0.indices, a0.data * scale_0), W.CSR(170, a1.indptr, a1.indices, a1.data * scale_k)]
    cp, ri = _window(170, 40)
    _check(sam, mats, cp, ri, steps)


def test_a_column_of_small_entries_among_ordinary_ones(sam):  # noqa: F811
    """One unknown's column is 1e-24 of the others (its squares vanish in FP32):
    solved in FP64, not rank deficient.  kappa is 1e24, so the map is compared
    where that column is no unknown, and has to be finite elsewhere."""
    import torch

    a0, a1 = _pair(170, 0.2, 3)
    data = np.where(a1.indices == 90, 1e-24, 1.0) * a1.data
    cp, ri = _window(170, 40)
    with sam.Handle() as h:
        S = h.sam_pattern_from_csc(170, torch.from_numpy(cp).cuda(), torch.from_numpy(ri).cuda())
        st = torch.empty(170, dtype=torch.int32, device="cuda")
        _, _, v = h.sam_build(sam.Csr.from_host(W.CSR(170, a1.indptr, a1.indices, data)), sam.Csr.from_host(a0), S, "fp32r",
                              1, col_status=st)
        h.sam_sync()
        solved64 = h.sam_refine_stats()[2]
        S.destroy()
    holds = (ri.reshape(170, 40) == 90).any(1)
    assert not st.cpu().numpy().any() and bool(torch.isfinite(v).all())
    assert solved64 == holds.sum()
