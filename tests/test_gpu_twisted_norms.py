"""Twisted solves in FP16/FP32 storage add the norms of alpha and beta over the sites in FP64.

At kappa = 3000 (no clover term, 2 kappa mu = 1) the squares of w = M M^dag r
are about 2e37 a site: within FP32 (3.4e38), but not summed over a tile of 128
sites.  A sum that leaves FP32 anywhere gives alpha = 0, and the first
iteration then adds nothing.  Bounds on x after it, against FP64: a handful of
roundings of the storage per component and one of alpha, 20 x 2^-24 in FP32
and 8 x 2^-11 in FP16 (the gate of the operator).
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


@pytest.mark.parametrize("prec,tol", [("fp32", 20 * 2.0 ** -24), ("fp16", 8 * 2.0 ** -11)])
@pytest.mark.parametrize("shape", [None, "0", "1"])
def test_tile_sums_beyond_fp32(lq, monkeypatch, prec, tol, shape):
    dims, nrhs, kappa = (8, 8, 8, 8), 3, 3000.0
    U = inputs.gauge_field(dims, 0.4, seed=21)
    b = inputs.spinor_field(dims, seed=22, nrhs=nrhs)
    lat = lq.lattice_create(dims)
    try:
        gid = lq.gauge_upload(lat, U)
        dp = lq.dirac_params(kappa, 0.0, mu=0.5 / kappa)
        ref, _, _ = lq.cg_solve(lat, gid, dp, lq.solver_params(tol=1e-6, maxiter=1, precision="fp64"), b, nrhs=nrhs)
        if shape is not None:
            monkeypatch.setenv("LQCD_HOP_NR", shape)
        x, info, _ = lq.cg_solve(lat, gid, dp, lq.solver_params(tol=1e-6, maxiter=1, precision=prec), b, nrhs=nrhs)
    finally:
        lq.lattice_destroy(lat)
    assert [i["iters_inner"] for i in info] == [1] * nrhs
    for j in range(nrhs):
        assert np.linalg.norm(x[j] - ref[j]) <= tol * np.linalg.norm(ref[j])
