"""CG on meshes large enough for the plane kernels (mf_plane.cuh): FP32 from 304 tiles, double-float
from 2048, with tile counts that leave the last FP32 CTA one tile past the end."""
import numpy as np
import pytest
import torch

import paper_2609_04534_gb300 as mf
from paper_2609_04534_gb300 import inputs
from tests._gpu import SHEAR_A, DevOp, rel_max
from tests.test_gpu_cg import consistent, solve

pytestmark = pytest.mark.gpu


def one_step(d, b, variant):
    """alpha of the first CG iteration from x = 0: x = alpha b"""
    mf.mf_operator_set_variant(d.op, variant)
    x = torch.empty_like(b)
    ws = torch.empty(mf.mf_cg_workspace_bytes(d.op, 0), dtype=torch.uint8, device="cuda")
    mf.mf_cg_solve(d.op, b.data_ptr(), x.data_ptr(), 0.0, 1, 0, ws.data_ptr(), ws.numel(), allow_not_converged=True)
    return float(torch.dot(x.double(), b.double()) / torch.dot(b.double(), b.double()))


def test_pairing_of_one_large_and_many_small_terms():
    """FP32, Q5, sheared, a mass term that outweighs the rest: u at the Gauss points of every cell
    (mirrored from cell to cell, so that u is continuous) is such that in every plane one point's term of
    <p, A p> is large and each other one just below half an ulp of it.  A plain sum over the
    plane drops up to 35 of them (1e-6 on average over the mirror images); a sum that drops only
    those of one row of n = 6 points agrees with the pencil kernel, which has the large ones in one
    pencil and drops none, within (n - 1) 2^-24."""
    k, dims = 5, (28, 27, 13)
    # a large term is 1.01 times a power of two, so that half an ulp of it is 0.99 2^-24 of it
    mass = 1.01 * 2.0**50 * np.prod(dims) / np.linalg.det(SHEAR_A)
    n = k + 1
    inner = np.polynomial.legendre.Legendre.basis(k).deriv().roots().real
    nodes = (np.concatenate([[-1.0], np.sort(inner), [1.0]]) + 1) / 2
    q, w = np.polynomial.legendre.leggauss(n)
    q, w = (q + 1) / 2, w / 2
    S = np.array([[np.prod([(x - nodes[m]) / (nodes[i] - nodes[m]) for m in range(n) if m != i]) for i in range(n)]
                  for x in q])
    small = 0.9 * 2.0**-24
    term = np.full((n, n, n), small)  # [z][y][x]
    term[:, 0, 0] = 1.0
    u = np.sqrt(term / (w[:, None, None] * w[:, None] * w))
    Si = np.linalg.inv(S)
    a = np.einsum("zc,yb,xa,cba->zyx", Si, Si, Si, u)  # nodal values

    def index(cells):  # local index of every global node, mirrored in odd cells
        node = np.arange(cells * k + 1)
        c, i = np.minimum(node // k, cells - 1), node - np.minimum(node // k, cells - 1) * k
        return np.where(c % 2 == 0, i, k - i)

    ix, iy, iz = (index(c) for c in dims)
    d = DevOp(*dims, k, "shear", mf.MF_HELMHOLTZ, mass, mf.MF_FP32, 0)
    b = d.native_from_unique(a[np.ix_(iz, iy, ix)].reshape(-1))
    plane, pencil = one_step(d, b, 0), one_step(d, b, 1)
    d.close()
    assert abs(plane / pencil - 1.0) <= (n - 1) * 2.0**-24, plane / pencil - 1.0


FP32, FP64 = mf.MF_FP32, mf.MF_FP64
CASES = ([(FP32, k, (28, 27, 13), g) for k in range(1, 6) for g in ("curved", "shear")] +
         [(FP32, k, (28, 27, 13), "cart") for k in (2, 6)] +
         [(FP64, 1, (44, 43, 33), g) for g in ("cart", "curved", "shear")] +
         [(FP64, 2, (44, 43, 33), g) for g in ("cart", "shear")])


@pytest.mark.parametrize("prec,k,dims,geom", CASES)
def test_split_forms_match_the_pencil_kernels_and_the_assembled_form(prec, k, dims, geom):
    """Six iterations: the split-dual forms (with the direction formed by its own kernel, and by the
    apply at load) on plane kernels, the same on pencil kernels, and the assembled form give the same
    residuals and iterate up to the rounding of the scalars, whose effect grows by less than an order
    per iteration; iterates stay consistent."""
    for kind, bc in ((mf.MF_LAPLACE, 1), (mf.MF_HELMHOLTZ, 0)):
        d = DevOp(*dims, k, geom, kind, 1.0, prec, bc)
        b = d.native_from_unique(inputs.random_unique(*dims, k, 23))
        its, tol = 6, 1e-4 if prec == FP32 else 1e-11
        mf.mf_operator_set_variant(d.op, 0)
        runs = [solve(d, b, 0.0, its, 0, hist_cap=its + 2, cg_form=f)
                for f in (mf.MF_CG_SPLIT_DUAL, mf.MF_CG_SPLIT_DUAL_FUSED, mf.MF_CG_ASSEMBLED)]
        mf.mf_operator_set_variant(d.op, 1)
        runs += [solve(d, b, 0.0, its, 0, hist_cap=its + 2, cg_form=f)
                 for f in (mf.MF_CG_SPLIT_DUAL, mf.MF_CG_SPLIT_DUAL_FUSED)]
        x0, st0, h0 = runs[0]
        assert st0["iterations"] == its and consistent(d, x0)
        for x, st, h in runs[1:]:
            assert st["iterations"] == its and consistent(d, x)
            np.testing.assert_allclose(h[:its + 1], h0[:its + 1], rtol=tol, atol=0)
            assert rel_max(d.unique_from_native(x), d.unique_from_native(x0)) <= tol
        d.close()
