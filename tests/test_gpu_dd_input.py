"""Conversion of double inputs in the double-float apply: mantissas whose leading 24 bits round up
into the next binade, just below and above powers of two, magnitudes on both sides of the window
that is converted without branches (2^-74), zeros, mixed signs -- against the FP64 oracle at the
library's FP64 contract (1e-12, relative max-norm), which a misplaced carry (an error of 2^-24 of one
value) exceeds by four orders."""
import numpy as np
import pytest

import paper_2609_04534_gb300 as mf
from tests._gpu import DevOp, oracle_op, rel_max

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("k", [1, 2, 3, 4, 6, 7, 8])
@pytest.mark.parametrize("geom", ["cart", "curved"])
@pytest.mark.parametrize("e", [-80, -74, 0, 60])
def test_input_conversion_edges(oracle, k, geom, e):
    dims = (5, 4, 3) if k <= 5 else (3, 2, 3)
    d = DevOp(*dims, k, geom, mf.MF_HELMHOLTZ, 1.0, mf.MF_FP64, 0)
    mf.mf_operator_set_variant(d.op, 1)  # a double-float variant at every degree
    o = oracle_op(oracle, *dims, k, geom, 1.0, 0)
    rng = np.random.default_rng(k)
    n = d.n_unique
    r = rng.integers(1, 2**30, n).astype(np.float64) * 2.0**-52
    x = np.where(rng.random(n) < 0.5, 2.0 - r, 1.0 + r) * np.where(rng.random(n) < 0.5, -1.0, 1.0)
    x[rng.random(n) < 0.1] = 0.0
    x *= 2.0**e
    y = d.unique_from_native(d.apply(d.native_from_unique(x)))
    assert rel_max(y, o.apply(x)) <= 1e-12
    d.close()
