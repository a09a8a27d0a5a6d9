"""A solve's last FP64 residual is that of the full lattice which ends it.

A right-hand side whose recursion has reached the target is closed on that
residual instead of on an FP64 update of its own.  With a small inner_tol no
update comes before, the residual of an FP16 or FP32 recursion is then smaller
than the true one and the closing check sends the solve back; with the default
it passes.  Both in each loop of the solver: captured (small), eager
(16^3 x 32 x 16 right-hand sides), batched, and with a mix of right-hand sides
that finish far apart, at once (zero) and never (maxiter).
"""
import numpy as np
import pytest

import oracle
from paper_2503_16994_gb300 import inputs

pytestmark = pytest.mark.gpu

CASES = [("fp64", 0.0), ("fp32", 0.0), ("fp32", 1e-14), ("fp16", 0.0), ("fp16", 1e-14)]


@pytest.fixture(scope="module")
def lq():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__
    __graft_entry__.build()
    from paper_2503_16994_gb300 import lqcd
    return lqcd


@pytest.mark.parametrize("prec,inner", CASES)
def test_small(lq, prec, inner):
    dims, tol, kappa, csw = (4, 6, 4, 8), 1e-10, 0.125, 1.2
    U = inputs.gauge_field(dims, 0.3, seed=301)
    b = inputs.spinor_field(dims, seed=302, nrhs=4)
    b[1] *= 1e-6  # the criterion is relative
    b[2] = 0.0
    b[3] = 0.0  # a point
    b[3].reshape(-1)[0] = 1.0
    lat = lq.lattice_create(dims)
    try:
        gid = lq.gauge_upload(lat, U)
        p = lq.dirac_params(kappa, csw)
        x, info, rc = lq.cg_solve(lat, gid, p, lq.solver_params(tol=tol, maxiter=20000, precision=prec,
                                                                inner_tol=inner), b, nrhs=4)
        _, short, rc_short = lq.cg_solve(lat, gid, p, lq.solver_params(tol=tol, maxiter=5, precision=prec,
                                                                       inner_tol=inner), b, nrhs=4)
    finally:
        lq.lattice_destroy(lat)
    assert rc == lq.OK, info
    assert not np.any(x[2])
    for j in (0, 1, 3):
        r = b[j] - oracle.dirac(dims, U, kappa, csw, x[j])
        got = np.linalg.norm(r) / np.linalg.norm(b[j])
        assert got <= tol and abs(got - info[j]["true_resid"]) <= 1e-14
    assert rc_short == lq.ENOCONV
    assert [s["status"] for s in short] == [lq.ENOCONV, lq.ENOCONV, lq.OK, lq.ENOCONV]


@pytest.mark.parametrize("prec,inner", CASES[1:])
def test_large(lq, prec, inner):
    dims, nrhs, tol = (16, 16, 16, 32), 16, 1e-9
    U = inputs.gauge_field(dims, 0.3, seed=303)
    b = np.concatenate([inputs.spinor_field(dims, seed=304, nrhs=2)] * (nrhs // 2))
    lat = lq.lattice_create(dims)
    try:
        gid = lq.gauge_upload(lat, U)
        p = lq.dirac_params(0.12, 1.2)
        x, info, rc = lq.cg_solve(lat, gid, p, lq.solver_params(tol=tol, maxiter=20000, precision=prec,
                                                                inner_tol=inner), b, nrhs=nrhs)
        assert rc == lq.OK, info
        for j in (0, 1, nrhs - 1):
            r = b[j] - lq.dirac_apply(lat, gid, p, x[j])
            got = np.linalg.norm(r) / np.linalg.norm(b[j])
            assert got <= tol and abs(got - info[j]["true_resid"]) <= 1e-13
    finally:
        lq.lattice_destroy(lat)


@pytest.mark.parametrize("prec,inner", CASES)
def test_batch(lq, prec, inner):
    sizes = [((4, 4, 4, 4), 0.2, 0.11), ((6, 4, 4, 8), 0.4, 0.125)]
    tol, lats, jobs = 1e-10, [], []
    try:
        for k, (dims, eps, kappa) in enumerate(sizes):
            lats.append(lq.lattice_create(dims))
            gid = lq.gauge_upload(lats[-1], inputs.gauge_field(dims, eps, seed=305 + k))
            jobs.append((lats[-1], gid, lq.dirac_params(kappa, 1.2), (1, 0, 2, 3), dims[3]))
        corrs, infos, statuses, rc = lq.pion_corr_batch(
            jobs, lq.solver_params(tol=tol, maxiter=20000, precision=prec, inner_tol=inner))
        assert rc == lq.OK and all(i["true_resid"] <= tol for info in infos for i in info)
        for k, (dims, eps, kappa) in enumerate(sizes):
            ref, *_ = oracle.pion(dims, inputs.gauge_field(dims, eps, seed=305 + k), kappa, 1.2, (1, 0, 2, 3),
                                  tol=1e-13)
            assert np.all(np.abs(corrs[k] - ref) <= 1e-8 * np.abs(ref))
    finally:
        for l in lats:
            lq.lattice_destroy(l)
