"""Launch variant 0 -- by degree, path, precision and mesh size a plane kernel or a pencil
configuration -- runs the pencil kernels' arithmetic: the split apply is bitwise that of launch
variants 1 and 2 on small and ragged meshes, and on meshes large enough for the plane kernels with
odd tile counts (an FP32 CTA takes two tiles, so the last one covers a tile past the end)."""
import pytest
import torch

import paper_2609_04534_gb300 as mf
from paper_2609_04534_gb300 import inputs
from tests._gpu import DevOp

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("k", range(1, 9))
@pytest.mark.parametrize("geom", ["cart", "shear", "curved"])
@pytest.mark.parametrize("dims", [(1, 1, 1), (4, 4, 2), (9, 4, 2), (5, 6, 3)])
def test_plane_kernels_equal_pencil_kernels(k, geom, dims):
    for prec, kind, bc in ((mf.MF_FP32, mf.MF_LAPLACE, 0), (mf.MF_FP32, mf.MF_HELMHOLTZ, 1),
                           (mf.MF_FP64, mf.MF_LAPLACE, 1), (mf.MF_FP64, mf.MF_HELMHOLTZ, 0)):
        d = DevOp(*dims, k, geom, kind, 1.0, prec, bc)
        x = d.native_from_unique(inputs.random_unique(*dims, k, 17))
        mf.mf_operator_set_variant(d.op, 0)
        y0 = d.apply(x, split=True)
        assert bool(torch.isfinite(y0).all())  # every lane is written
        for v in (1, 2):
            mf.mf_operator_set_variant(d.op, v)
            y = d.apply(x, split=True)
            torch.cuda.synchronize()
            assert torch.equal(y, y0), (prec, kind, bc, v)
        d.close()


# 7 x 7 x 7 tiles (FP32 planes from 304 tiles); 11 x 11 x 17 (double-float planes from 2048)
@pytest.mark.parametrize("prec,k,dims", [(mf.MF_FP32, k, (28, 27, 13)) for k in range(1, 7)] +
                         [(mf.MF_FP64, k, (44, 43, 33)) for k in (1, 2)])
@pytest.mark.parametrize("geom", ["cart", "shear", "curved"])
def test_plane_kernels_on_meshes_that_use_them(prec, k, dims, geom):
    for kind, bc in ((mf.MF_LAPLACE, 1), (mf.MF_HELMHOLTZ, 0)):
        d = DevOp(*dims, k, geom, kind, 1.0, prec, bc)
        x = d.native_from_unique(inputs.random_unique(*dims, k, 18))
        mf.mf_operator_set_variant(d.op, 0)
        y0 = d.apply(x, split=True)
        assert bool(torch.isfinite(y0).all())
        mf.mf_operator_set_variant(d.op, 1)
        y = d.apply(x, split=True)
        torch.cuda.synchronize()
        assert torch.equal(y, y0), (kind, bc)
        d.close()
