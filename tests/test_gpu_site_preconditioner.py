"""GPU solves with the even site term divided out, where that term matters.

The solver iterates on Dhat A_ee^-1.  Cases: no clover term (A = 1), a strong
one on a rough field (site blocks far from 1), twisted mass (its inverse has
two block pairs), open and SF boundaries (identity blocks and boundary terms),
one site per warp's end (2^4) and a partly filled block, in every precision,
from zero and from a guess.  The residual is the oracle's, <= tol; the
reported one agrees with it.
"""
import numpy as np
import pytest

import oracle
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


CASES = [((2, 2, 2, 2), 0.3, 0.12, 0.0, 0.0, "periodic"), ((6, 4, 2, 10), 0.8, 0.115, 2.2, 0.0, "periodic"),
         ((6, 4, 2, 10), 0.6, 0.12, 1.9, 0.1, "periodic"), ((4, 4, 6, 6), 0.5, 0.12, 1.7, 0.0, "open"),
         ((4, 4, 6, 6), 0.5, 0.12, 1.7, 0.0, "sf")]


@pytest.mark.parametrize("dims,eps,kappa,csw,mu,bc", CASES)
@pytest.mark.parametrize("prec", ["fp64", "fp32", "fp16"])
@pytest.mark.parametrize("guess", [False, True])
def test_solve(lq, dims, eps, kappa, csw, mu, bc, prec, guess):
    nrhs, tol = 3, 1e-11
    U = inputs.gauge_field(dims, eps, seed=221)
    b = inputs.spinor_field(dims, seed=222, nrhs=nrhs)
    x0 = 0.3 * inputs.spinor_field(dims, seed=223, nrhs=nrhs)
    lat = lq.lattice_create(dims)
    try:
        gid = lq.gauge_upload(lat, U)
        x, info, rc = lq.cg_solve(lat, gid, lq.dirac_params(kappa, csw, mu=mu, bc=bc, cF=1.2),
                                  lq.solver_params(tol=tol, maxiter=20000, precision=prec), b, nrhs=nrhs,
                                  x=x0 if guess else None, guess=guess)
    finally:
        lq.lattice_destroy(lat)
    assert rc == lq.OK, info
    for j in range(nrhs):
        if bc == "open":
            r = b[j] - oracle.dirac_open(dims, U, kappa, csw, 1.2, x[j])
        elif bc == "sf":
            r = b[j] - oracle.dirac_sf(dims, U, kappa, csw, 1.2, x[j])
        else:
            r = b[j] - oracle.dirac_tm(dims, U, kappa, csw, mu, x[j])
        got = np.linalg.norm(r) / np.linalg.norm(b[j])
        assert got <= tol and abs(got - info[j]["true_resid"]) <= 1e-14
