"""CG on every shape of the hopping kernels.

The solver's hops (self + H, with the norm of alpha, and self + clover H of the
adjoint, with that of beta) are built for each shape: right-hand sides per
thread (1 to 3), paired (0), prefetching (-2, -4, -8), staged (12, 13) and tile
(20, 21), twisted scalar and paired.  Five right-hand sides (a half-empty last
pair or triple) on 240 sites of a parity (a partly filled last tile), all shapes
forced in turn.  The residual is the oracle's; a wrong norm would show as other
iterations than the scalar shape's: FP16 shapes give the same bits, FP32 ones
round differently, which moves a stop by at most a few iterations.
"""
import numpy as np
import pytest

import oracle
from paper_2503_16994_gb300 import inputs

pytestmark = pytest.mark.gpu
DIMS, NRHS, KAPPA, CSW, TOL = (6, 4, 2, 10), 5, 0.125, 1.4, 1e-10


@pytest.fixture(scope="module")
def lq():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__
    __graft_entry__.build()
    from paper_2503_16994_gb300 import lqcd
    return lqcd


def solves(lq, monkeypatch, prec, mu, shapes):
    """{shape: (x, iterations)}; shape = (right-hand-side code, groups per block)"""
    U = inputs.gauge_field(DIMS, 0.4, seed=801)
    b = inputs.spinor_field(DIMS, seed=802, nrhs=NRHS)
    out = {}
    lat = lq.lattice_create(DIMS)
    try:
        gid = lq.gauge_upload(lat, U)
        for nr, gpb in shapes:
            monkeypatch.setenv("LQCD_HOP_NR", str(nr))
            monkeypatch.setenv("LQCD_HOP_GPB", str(gpb))
            x, info, rc = lq.cg_solve(lat, gid, lq.dirac_params(KAPPA, CSW, mu=mu),
                                      lq.solver_params(tol=TOL, maxiter=2000, precision=prec), b, nrhs=NRHS)
            assert rc == lq.OK, (nr, gpb, info)
            for j in range(NRHS):
                r = b[j] - oracle.dirac_tm(DIMS, U, KAPPA, CSW, mu, x[j])
                assert np.linalg.norm(r) <= 1.001 * TOL * np.linalg.norm(b[j]), (nr, gpb, j)
            out[nr, gpb] = x, [i["iters_inner"] for i in info]
    finally:
        lq.lattice_destroy(lat)
    return out


def check(out, same_bits):
    x0, its0 = out[1, 1]
    for shape, (x, its) in out.items():
        if same_bits:
            assert its == its0 and np.array_equal(x, x0), shape
        else:
            assert np.max(np.abs(np.subtract(its, its0))) <= 3, (shape, its, its0)


@pytest.mark.parametrize("prec", ["fp32", "fp16"])
def test_untwisted(lq, monkeypatch, prec):
    shapes = [(1, 1), (2, 1), (3, 1), (3, 2), (0, 1), (0, 2), (-2, 1), (-4, 2), (-8, 1)]
    if prec == "fp16":
        shapes += [(12, 1), (12, 3), (13, 1), (20, 3), (21, 1)]
    check(solves(lq, monkeypatch, prec, 0.0, shapes), prec == "fp16")


@pytest.mark.parametrize("prec", ["fp32", "fp16"])
def test_twisted(lq, monkeypatch, prec):
    check(solves(lq, monkeypatch, prec, 0.07, [(1, 1), (1, 3), (0, 1), (0, 3)]), prec == "fp16")
