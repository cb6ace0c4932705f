"""Chunk lengths of mf_cg_solve: any length gives the same solve, the largest an int holds included
(a chunk stops at maxit)."""
import pytest
import torch

import paper_2609_04534_gb300 as mf
from paper_2609_04534_gb300 import inputs
from tests._gpu import DevOp, rel_max

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("chunk", [1, 7, 10**9, 2**31 - 1])
def test_chunk_length_does_not_change_the_solve(chunk):
    d = DevOp(6, 6, 6, 3, "curved", mf.MF_LAPLACE, 1.0, mf.MF_MIXED, 1)
    b = d.native_from_unique(inputs.random_unique(6, 6, 6, 3, 9))
    ws = torch.empty(mf.mf_cg_workspace_bytes(d.op, 1), dtype=torch.uint8, device="cuda")
    out = []
    for c in (0, chunk):
        x = torch.empty_like(b)
        st = mf.mf_cg_solve(d.op, b.data_ptr(), x.data_ptr(), 1e-10, 1500, 1, ws.data_ptr(), ws.numel(), chunk_iterations=c)
        out.append((d.unique_from_native(x), st))
    assert out[0][1]["outer_iterations"] >= 3  # past the chunks that are launched directly
    assert out[1][1]["iterations"] == out[0][1]["iterations"]
    assert rel_max(out[1][0], out[0][0]) == 0.0
    d.close()
