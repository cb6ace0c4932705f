"""CG on meshes large enough for the plane kernels (mf_plane.cuh)."""
import numpy as np
import pytest
import torch

import paper_2609_04534_gb300 as mf
from tests._gpu import SHEAR_A, DevOp

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
