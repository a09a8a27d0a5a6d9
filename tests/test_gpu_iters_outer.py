"""iters_outer counts the FP64 residual that closes a solve.

Solves whose recursion reaches the target without an update before (FP64, and
a small inner_tol with a loose target) report exactly that one; a zero
right-hand side none.  In the captured, the batched and the eager loop.
"""
import numpy as np
import pytest

from paper_2503_16994_gb300 import inputs

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def lq():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__
    __graft_entry__.build()
    from paper_2503_16994_gb300 import lqcd
    return lqcd


@pytest.mark.parametrize("prec,tol", [("fp64", 1e-10), ("fp32", 1e-3), ("fp16", 1e-1)])
@pytest.mark.parametrize("dims,nrhs", [((4, 4, 4, 8), 3), ((16, 16, 16, 32), 16)])
def test_solve(lq, prec, tol, dims, nrhs):
    if prec == "fp64" and nrhs == 16:
        pytest.skip("the eager loop is the same for every precision; FP64 there takes seconds")
    b = np.concatenate([inputs.spinor_field(dims, seed=402, nrhs=1)] * nrhs)
    b[1] = 0.0
    lat = lq.lattice_create(dims)
    try:
        gid = lq.gauge_upload(lat, inputs.gauge_field(dims, 0.3, seed=401))
        _, info, rc = lq.cg_solve(lat, gid, lq.dirac_params(0.12, 1.2),
                                  lq.solver_params(tol=tol, precision=prec, inner_tol=1e-14), b, nrhs=nrhs)
    finally:
        lq.lattice_destroy(lat)
    assert rc == lq.OK
    assert [i["iters_outer"] for i in info] == [1, 0] + [1] * (nrhs - 2)


def test_batch(lq):
    dims = (4, 4, 4, 6)
    lat = lq.lattice_create(dims)
    try:
        gid = lq.gauge_upload(lat, inputs.gauge_field(dims, 0.3, seed=403))
        _, infos, _, rc = lq.pion_corr_batch([(lat, gid, lq.dirac_params(0.12, 1.2), (0, 0, 0, 0), 6)],
                                             lq.solver_params(tol=1e-10, precision="fp64"))
    finally:
        lq.lattice_destroy(lat)
    assert rc == lq.OK and [i["iters_outer"] for i in infos[0]] == [1] * 12
