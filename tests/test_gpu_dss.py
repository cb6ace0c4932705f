"""The duplicate summation (mf_dss) and the average of copies (mf_make_consistent) against
dimension-split sweeps in numpy: the copies of a node summed pairwise along x, then y, then z,
each sum one addition in the vector's own type.  Every sum is the same single rounding in the
same order, so the results are equal bit for bit (tolerance 0)."""
import numpy as np
import pytest
import torch

import paper_2609_04534_gb300 as mf
from tests._gpu import DevOp

pytestmark = pytest.mark.gpu

# one cell; one cell thick in each direction; exactly one tile (4x4x2); a tile plus one cell in
# every direction; ragged tiles in every direction
DIMS = [(1, 1, 1), (9, 1, 2), (1, 6, 5), (4, 4, 2), (5, 5, 3), (9, 6, 5)]


def sweeps(y, k, avg, bc):
    """y: [cz, cy, cx, k, j, i]."""
    y = y.copy()
    for cell, loc in ((2, 5), (1, 4), (0, 3)):
        c, l = np.moveaxis(y, (cell, loc), (0, 1)), k
        s = c[:-1, l] + c[1:, 0]
        if avg:
            s = s * y.dtype.type(0.5)
        c[:-1, l] = s
        c[1:, 0] = s
    if bc and not avg:
        for cell, loc in ((2, 5), (1, 4), (0, 3)):
            c = np.moveaxis(y, (cell, loc), (0, 1))
            c[0, 0] = 0
            c[-1, k] = 0
    return y


@pytest.mark.parametrize("k", range(1, 9))
@pytest.mark.parametrize("dims", DIMS)
def test_dss_equals_dimension_split_sweeps(k, dims):
    nx, ny, nz = dims
    for prec, bc in ((mf.MF_FP64, 0), (mf.MF_FP64, 1), (mf.MF_FP32, 1)):
        d = DevOp(nx, ny, nz, k, "cart", mf.MF_LAPLACE, 1.0, prec, bc)
        nt = np.float32 if prec == mf.MF_FP32 else np.float64
        y0 = np.random.default_rng(k).standard_normal((nz, ny, nx, k + 1, k + 1, k + 1)).astype(nt)
        can = torch.as_tensor(y0.ravel(), device="cuda")
        for avg in (False, True):
            nat = torch.empty(d.n_native, dtype=d.dtype, device="cuda")
            mf.mf_to_native(d.op, can.data_ptr(), nat.data_ptr())
            (mf.mf_make_consistent if avg else mf.mf_dss)(d.op, nat.data_ptr())
            got = d.canonical_from_native(nat).astype(nt).reshape(y0.shape)
            assert np.array_equal(got, sweeps(y0, k, avg, bc)), (prec, bc, avg)
        d.close()
