"""Residual update of large batches: four 128-site tiles per block.

26 right-hand sides on 12^3 x 24 are 26 x 162 tiles (the last block of each has
two), two are 324 and take one tile per block.  The sums are formed in the
same order, so in FP16, where every kernel shape stores the same bits, the
solutions are equal; in FP32 and FP64 the residual is the library's own D.
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


@pytest.mark.parametrize("prec", ["fp16", "fp32", "fp64"])
def test_many_tiles(lq, prec):
    dims, nrhs, tol = (12, 12, 12, 24), 26, 1e-10
    U = inputs.gauge_field(dims, 0.3, seed=401)
    two = inputs.spinor_field(dims, seed=402, nrhs=2)
    b = np.concatenate([two] * (nrhs // 2))
    lat = lq.lattice_create(dims)
    try:
        gid = lq.gauge_upload(lat, U)
        p, sp = lq.dirac_params(0.12, 1.2), lq.solver_params(tol=tol, maxiter=5000, precision=prec)
        x, info, rc = lq.cg_solve(lat, gid, p, sp, b, nrhs=nrhs)
        assert rc == lq.OK, info
        if prec == "fp16":
            x2, info2, rc2 = lq.cg_solve(lat, gid, p, sp, two, nrhs=2)
            assert rc2 == lq.OK
            for j in range(nrhs):
                assert info[j]["iters_inner"] == info2[j % 2]["iters_inner"]
                assert np.array_equal(x[j], x2[j % 2])
        for j in (0, 1, nrhs - 1):
            r = b[j] - lq.dirac_apply(lat, gid, p, x[j])
            assert np.linalg.norm(r) <= tol * np.linalg.norm(b[j])
    finally:
        lq.lattice_destroy(lat)
