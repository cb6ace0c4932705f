"""Breakdown of CG in the split-dual update, which finds <p, A p> <= 0 itself: an indefinite
operator (Helmholtz with a negative mass coefficient) on meshes whose update takes many CTAs.  The
solve stops with MF_ERR_BREAKDOWN and the iterate before it, bitwise that of a solve with maxit
iterations up to there, on every repetition; in a batch the other members are not touched."""
import re

import numpy as np
import pytest
import torch

import paper_2609_04534_gb300 as mf
from paper_2609_04534_gb300 import inputs
from tests._gpu import DevOp
from tests.test_gpu_serving import make_server, run

pytestmark = pytest.mark.gpu


def solve(d, b, maxit, ws, cg_form, mixed):
    """(x, iteration of the breakdown or None)"""
    x = torch.full((d.n_native,), float("nan"), dtype=d.dtype, device="cuda")
    try:
        st = mf.mf_cg_solve(d.op, b.data_ptr(), x.data_ptr(), 0.0, maxit, mixed, ws.data_ptr(), ws.numel(),
                            allow_not_converged=True, cg_form=cg_form)
        assert st["iterations"] == maxit
        return x, None
    except mf.MfError as e:
        assert e.code == mf.MF_ERR_BREAKDOWN, e
        return x, int(re.search(r"at iteration (\d+)", str(e)).group(1))


@pytest.mark.parametrize("dims,k,geom,prec,bc,mass", [
    ((13, 11, 9), 3, "curved", mf.MF_FP64, 1, -200.0),
    ((13, 11, 9), 2, "cart", mf.MF_FP64_DFMA, 1, -200.0),
    ((28, 27, 13), 2, "shear", mf.MF_FP32, 0, -200.0),
    ((9, 10, 11), 4, "cart", mf.MF_FP32, 0, -1000.0),
])
def test_breakdown_leaves_the_iterate_before_it(dims, k, geom, prec, bc, mass):
    d = DevOp(*dims, k, geom, mf.MF_HELMHOLTZ, mass, prec, bc)
    b = d.native_from_unique(inputs.random_unique(*dims, k, 3))
    ws = torch.empty(mf.mf_cg_workspace_bytes(d.op, 0), dtype=torch.uint8, device="cuda")
    for form in (mf.MF_CG_SPLIT_DUAL, mf.MF_CG_SPLIT_DUAL_FUSED):
        x, at = solve(d, b, 100, ws, form, 0)
        assert at is not None and at >= 1
        before, none = solve(d, b, at, ws, form, 0)
        assert none is None and bool(torch.isfinite(before).all())
        assert torch.equal(x, before)
        for _ in range(20):
            x, again = solve(d, b, 100, ws, form, 0)
            assert again == at and torch.equal(x, before)
    d.close()


@pytest.mark.parametrize("mixed", [0, 1])
def test_breakdown_of_batched_members(mixed):
    """Requests of one class: four break down, four do not; the latter equal their solves alone."""
    reqs = [dict(nx=13, ny=11, nz=8 + i, degree=3, geometry=mf.MF_AFFINE, kind=mf.MF_HELMHOLTZ,
                 mass_coeff=-200.0 if i % 2 else 1.0, rhs=mf.MF_RHS_RANDOM, seed=70 + i, mixed=mixed) for i in range(8)]
    for _ in range(3):
        sv, arena = make_server(slots=16)
        try:
            res, xs = run(sv, [mf.make_request(**p) for p in reqs])
        finally:
            mf.mf_server_destroy(sv)
        for i, r in enumerate(res):
            assert r["status"] == (mf.MF_ERR_BREAKDOWN if i % 2 else mf.MF_OK), (i, r)
    for i in (0, 2, 4, 6):
        sv, arena = make_server(slots=1, batching=-1)
        try:
            (r1,), (x1,) = run(sv, [mf.make_request(**reqs[i])])
        finally:
            mf.mf_server_destroy(sv)
        assert r1["iterations"] == res[i]["iterations"] and np.array_equal(x1, xs[i])
