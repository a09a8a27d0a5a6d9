"""GPU twisted mass on the scalar and the paired hopping kernels.

Both shapes, forced, with one to five right-hand sides (a half-empty last
pair) on ragged lattices (extents of 2, partly filled blocks), D and D^dag,
complex boundary phases: FP32 and FP16 against FP64 within the gates of the
untwisted operator (2e-6, 4e-3), and in FP16 the two shapes give the same
bits.  Solves past the small-batch rule run the FP64 set-up and final modes.
"""
import numpy as np
import pytest

import oracle
from paper_2503_16994_gb300 import inputs

pytestmark = pytest.mark.gpu
THETA = (np.exp(0.3j), 1, 1, -1)


@pytest.fixture(scope="module")
def lq():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__
    __graft_entry__.build()
    from paper_2503_16994_gb300 import lqcd
    return lqcd


def even(dims):
    lx, ly, lz, lt = dims
    t, z, y, x = np.meshgrid(np.arange(lt), np.arange(lz), np.arange(ly), np.arange(lx), indexing="ij")
    return ((x + y + z + t) % 2 == 0)[..., None, None]


def rel(a, b):
    return np.linalg.norm(a - b) / np.linalg.norm(b)


@pytest.mark.parametrize("dims", [(2, 2, 2, 2), (6, 4, 2, 10)])
@pytest.mark.parametrize("nrhs", [1, 2, 5])
@pytest.mark.parametrize("prec,tol", [("fp32", 2e-6), ("fp16", 4e-3)])
def test_shapes(lq, monkeypatch, dims, nrhs, prec, tol):
    U = inputs.gauge_field(dims, 0.4, seed=211)
    x = inputs.spinor_field(dims, seed=212, nrhs=nrhs) * even(dims)
    lat = lq.lattice_create(dims)
    try:
        gid = lq.gauge_upload(lat, U)
        dp = lq.dirac_params(0.13, 1.5, THETA, mu=-0.08)
        for dagger in (False, True):
            ref = lq.schur_apply(lat, gid, dp, x, precision="fp64", nrhs=nrhs, dagger=dagger)
            got = []
            for nr, gpb in ((1, 1), (0, 1), (0, 3)):
                monkeypatch.setenv("LQCD_HOP_NR", str(nr))
                monkeypatch.setenv("LQCD_HOP_GPB", str(gpb))
                got.append(lq.schur_apply(lat, gid, dp, x, precision=prec, nrhs=nrhs, dagger=dagger))
                monkeypatch.delenv("LQCD_HOP_NR")
                monkeypatch.delenv("LQCD_HOP_GPB")
            got.append(lq.schur_apply(lat, gid, dp, x, precision=prec, nrhs=nrhs, dagger=dagger))
            for g in got:
                for j in range(nrhs):
                    assert rel(g[j], ref[j]) <= tol
                if prec == "fp16":
                    assert np.array_equal(g, got[0])
    finally:
        lq.lattice_destroy(lat)


@pytest.mark.parametrize("prec", ["fp64", "fp16"])
def test_solve_past_the_small_batch_rule(lq, prec):
    dims, nrhs, mu = (8, 8, 8, 12), 5, 0.06  # 3072 sites x 5 right-hand sides
    U = inputs.gauge_field(dims, 0.3, seed=213)
    b = inputs.spinor_field(dims, seed=214, nrhs=nrhs)
    lat = lq.lattice_create(dims)
    try:
        gid = lq.gauge_upload(lat, U)
        x, info, rc = lq.cg_solve(lat, gid, lq.dirac_params(0.125, 1.3, THETA, mu=mu),
                                  lq.solver_params(tol=1e-11, maxiter=5000, precision=prec), b, nrhs=nrhs)
    finally:
        lq.lattice_destroy(lat)
    assert rc == lq.OK, info
    for j in (0, nrhs - 1):
        r = b[j] - oracle.dirac_tm(dims, U, 0.125, 1.3, mu, x[j], theta=THETA)
        assert np.linalg.norm(r) <= 1e-11 * np.linalg.norm(b[j])
