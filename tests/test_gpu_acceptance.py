"""A solve closed by its recursion meets the acceptance of one closed by an FP64 update.

An FP64 residual update stops a right-hand side at tol / 2.  A recursion that
says so has to be borne out by the FP64 residual of the full lattice at that
same line, whatever inner_tol lets the recursion drift by; the two residuals
agree to FP64 rounding (1e-14 of b).  Alone, batched, and served next to the
same request alone.
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


@pytest.mark.parametrize("prec", ["fp64", "fp32", "fp16"])
@pytest.mark.parametrize("inner", [0.0, 1e-2, 1e-3])
def test_residuals(lq, prec, inner):
    dims = (8, 8, 8, 12)
    lat = lq.lattice_create(dims)
    got = []
    try:
        gid = lq.gauge_upload(lat, inputs.gauge_field(dims, 0.35, seed=11))
        for seed in range(3):
            b = inputs.spinor_field(dims, seed=50 + seed, nrhs=8)
            for tol in (1e-6, 3e-8, 1e-10):
                _, info, rc = lq.cg_solve(lat, gid, lq.dirac_params(0.128, 1.4),
                                          lq.solver_params(tol=tol, precision=prec, inner_tol=inner), b, nrhs=8)
                assert rc == lq.OK, info
                got += [i["true_resid"] - 0.5 * tol for i in info]
        jobs = [(lat, gid, lq.dirac_params(k, 1.4), (0, 1, 2, 3), 12) for k in (0.12, 0.128)]
        _, infos, _, rc = lq.pion_corr_batch(jobs, lq.solver_params(tol=1e-8, precision=prec, inner_tol=inner))
        assert rc == lq.OK
        got += [i["true_resid"] - 0.5e-8 for info in infos for i in info]
    finally:
        lq.lattice_destroy(lat)
    assert max(got) <= 1e-14


@pytest.mark.parametrize("prec,inner", [("fp64", 0.0), ("fp32", 1e-3), ("fp16", 1e-3)])
def test_served_and_alone(lq, prec, inner):
    dims, tol, src = (6, 4, 4, 8), 1e-9, (1, 2, 3, 4)
    U = inputs.gauge_field(dims, 0.35, seed=12)
    dp, sp = lq.dirac_params(0.128, 1.4), lq.solver_params(tol=tol, precision=prec, inner_tol=inner)
    lat, srv = lq.lattice_create(dims), lq.serve_create(max_slots=1)
    try:
        corr, _, alone, rc = lq.pion_corr(lat, lq.gauge_upload(lat, U), dp, sp, src, dims=dims)
        assert rc == lq.OK
        ticket = lq.serve_submit(srv, lq.serve_gauge(srv, dims, U), dp, sp, src)
        rc, served, info, _ = lq.serve_poll(srv, ticket, dims[3], timeout_ms=60000)
        assert rc == lq.OK
    finally:
        lq.serve_destroy(srv)
        lq.lattice_destroy(lat)
    for i in alone + info:
        assert i["true_resid"] <= 0.5 * tol + 1e-14
    assert np.max(np.abs(served - corr)) <= 1e-7 * np.max(corr)  # both within tol / 2, amplified by |D^-1| < 50
