"""Accuracy of the apply kernels against the oracle's 64-bit arithmetic, by the relative L2
error over several inputs: not larger than with the full-length products (fma in mf_dd.cuh) and,
in FP32, with products contracted into sums, whose errors on these inputs are listed.  The
computation is deterministic; the margin covers the order of the CG scalars' 64-bit sums (1e-16 of
errors of 1e-14)."""
import numpy as np
import pytest
import torch

import paper_2609_04534_gb300 as mf
from paper_2609_04534_gb300 import inputs
from tests._gpu import DevOp, oracle_op

pytestmark = pytest.mark.gpu


def relative(pairs):
    num = sum(float(((a - b) ** 2).sum()) for a, b in pairs)
    return (num / sum(float((b ** 2).sum()) for _, b in pairs)) ** 0.5


def cg_error(oracle, geom, k):
    """x after four iterations of FP64 CG (double-float vectors), 10^3 cells, Laplace."""
    d = DevOp(10, 10, 10, k, geom, mf.MF_LAPLACE, 1.0, mf.MF_FP64, 1)
    o = oracle_op(oracle, 10, 10, 10, k, geom, 0.0, 1)
    ws = torch.empty(mf.mf_cg_workspace_bytes(d.op, 0), dtype=torch.uint8, device="cuda")
    pairs = []
    for seed in (5, 6, 7, 8):
        bu = inputs.random_unique(10, 10, 10, k, seed)
        b = d.native_from_unique(bu)
        x = torch.empty_like(b)
        mf.mf_cg_solve(d.op, b.data_ptr(), x.data_ptr(), 0.0, 4, 0, ws.data_ptr(), ws.numel(), allow_not_converged=True)
        ref, _ = o.cg(np.where(o.boundary_mask(), 0.0, bu), maxit=4, rtol=0.0)
        pairs.append((d.unique_from_native(x), ref))
    d.close()
    return relative(pairs)


def apply_error(oracle, geom, k, prec):
    """the apply, 11 x 9 x 10 cells, Laplace"""
    dims = (11, 9, 10)
    d = DevOp(*dims, k, geom, mf.MF_LAPLACE, 1.0, prec, 1)
    o = oracle_op(oracle, *dims, k, geom, 0.0, 1)
    pairs = []
    for seed in (5, 6, 7):
        xu = inputs.random_unique(*dims, k, seed)
        if prec == mf.MF_FP32:
            xu = xu.astype(np.float32).astype(np.float64)
        pairs.append((d.unique_from_native(d.apply(d.native_from_unique(xu))), o.apply(xu)))
    d.close()
    return relative(pairs)


# with full-length products everywhere
CG = {("cart", 4): 8.890e-15, ("cart", 6): 1.330e-14, ("cart", 7): 1.901e-14, ("curved", 4): 1.162e-14,
      ("shear", 4): 1.369e-14}
APPLY = {("curved", 2): 5.4001e-15, ("shear", 2): 7.2812e-15}


@pytest.mark.parametrize("geom,k", list(CG))
def test_cg_vectors_in_double_float_lose_nothing(oracle, geom, k):
    assert cg_error(oracle, geom, k) <= 1.01 * CG[geom, k]


@pytest.mark.parametrize("geom,k", list(APPLY))
def test_apply_with_truncated_input_loses_nothing(oracle, geom, k):
    assert apply_error(oracle, geom, k, mf.MF_FP64) <= 1.001 * APPLY[geom, k]


FP32 = {("cart", 2): 1.2651e-07, ("shear", 2): 1.3249e-07}  # one rounding per product and sum


@pytest.mark.parametrize("geom,k", list(FP32))
def test_fp32_products_go_into_sums_by_one_rounding(oracle, geom, k):
    assert apply_error(oracle, geom, k, mf.MF_FP32) <= 1.001 * FP32[geom, k]
