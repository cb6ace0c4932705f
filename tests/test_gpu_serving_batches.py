"""Requests of one class that arrive one after another share batched chunks."""
import time

import numpy as np
import pytest

import paper_2609_04534_gb300 as mf
from paper_2609_04534_gb300 import inputs
from tests.test_gpu_serving import make_server, run

pytestmark = pytest.mark.gpu


def test_staggered_requests_of_one_class_run_in_batches():
    """Eight FP64 requests (curved Q4, 16^3 cells; hundreds of iterations each, tens of milliseconds)
    submitted 3 ms apart overlap, and fall into step though the first ones start alone: more
    than half of all iterations come from batches, of at least two members; the solution of one of
    them is bitwise that of the request alone."""
    n, k = 16, 4
    reqs = [dict(nx=n, ny=n, nz=n, degree=k, geometry=mf.MF_CURVED_SIN, rhs=mf.MF_RHS_RANDOM, seed=90 + i, mixed=0,
                 rtol=1e-14, maxit=20000) for i in range(8)]
    sv, arena = make_server(slots=16)
    try:
        run(sv, [mf.make_request(**dict(reqs[0], maxit=20))])  # loads the kernels
        c0, m0 = mf.mf_server_batch_counts(sv)
        outs, tickets = [], []
        for p in reqs:
            outs.append(np.zeros(inputs.unique_count(n, n, n, k)))
            tickets.append(mf.mf_batch_submit(sv, mf.make_request(**p, x_out_ptr=outs[-1].ctypes.data)))
            time.sleep(0.003)
        mf.mf_server_drain(sv, 120.0)
        res = [mf.mf_batch_poll(sv, t) for t in tickets]
        c1, m1 = mf.mf_server_batch_counts(sv)
    finally:
        mf.mf_server_destroy(sv)
    assert all(r["status"] == mf.MF_OK for r in res), res
    assert 10 * (m1 - m0) >= 0.5 * sum(r["iterations"] for r in res), (c1 - c0, m1 - m0)
    assert m1 - m0 >= 2 * (c1 - c0)
    sv, arena = make_server(slots=1, batching=-1)
    try:
        (r1,), (x1,) = run(sv, [mf.make_request(**reqs[3])])
    finally:
        mf.mf_server_destroy(sv)
    assert r1["iterations"] == res[3]["iterations"] and np.array_equal(x1, outs[3])


@pytest.mark.parametrize("geometry,k", [(mf.MF_AFFINE, 1), (mf.MF_AFFINE, 2), (mf.MF_AFFINE, 3), (mf.MF_CURVED_SIN, 1)])
def test_batched_plane_kernels_match_solo_solves(geometry, k):
    """Mixed requests whose FP32 inner CG runs on plane kernels at any size (Cartesian of degrees 1
    to 3, general of degree 1), ragged meshes with odd tile counts, in one batch: bitwise the solutions
    of the requests alone."""
    reqs = [dict(nx=5 + 2 * i, ny=7, nz=3 + i, degree=k, geometry=geometry, rhs=mf.MF_RHS_RANDOM, seed=40 + i, mixed=1)
            for i in range(6)]
    sv, arena = make_server(slots=16)
    try:
        res, xs = run(sv, [mf.make_request(**p) for p in reqs])
        chunks, members = mf.mf_server_batch_counts(sv)
    finally:
        mf.mf_server_destroy(sv)
    assert members >= 2 * chunks > 0
    for p, r, x in zip(reqs, res, xs):
        sv, arena = make_server(slots=1, batching=-1)
        try:
            (r1,), (x1,) = run(sv, [mf.make_request(**p)])
        finally:
            mf.mf_server_destroy(sv)
        assert r["status"] == r1["status"] == mf.MF_OK and r1["iterations"] == r["iterations"]
        assert np.array_equal(x1, x), p
