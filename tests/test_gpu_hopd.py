"""GPU FP64 operator on both sides of the rule that gives small batches to the kernel with 16 threads per site.

At most 12288 sites of a parity times right-hand sides run there (the last
size of its range, one with a partly filled block, extents of 2), larger ones
on the kernel with one thread per site.  D and D^dag with complex boundary
phases, twisted and not, against the oracle within 1e-13 (about 100 FP64
roundings per component); the two kernels store the same bits; solves in FP64
on the small side go through its norm-computing modes.
"""
import numpy as np
import pytest

import oracle
from paper_2503_16994_gb300 import inputs

pytestmark = pytest.mark.gpu
THETA = (np.exp(0.3j), 1, np.exp(-0.7j), -1)


@pytest.fixture(scope="module")
def lq():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__
    __graft_entry__.build()
    from paper_2503_16994_gb300 import lqcd
    return lqcd


@pytest.mark.parametrize("dims", [(2, 2, 2, 2), (2, 6, 2, 6), (6, 4, 10, 2), (8, 12, 8, 32), (8, 12, 10, 26)])
@pytest.mark.parametrize("mu", [0.0, 0.07])
def test_dirac_both_sides(lq, dims, mu):
    U = inputs.gauge_field(dims, 0.4, seed=95)
    psi = inputs.spinor_field(dims, seed=96)
    lat = lq.lattice_create(dims)
    try:
        gid = lq.gauge_upload(lat, U)
        for dagger in (False, True):
            got = lq.dirac_apply(lat, gid, lq.dirac_params(0.13, 1.5, THETA, mu=mu), psi, dagger=dagger)
            want = oracle.dirac_tm(dims, U, 0.13, 1.5, mu, psi, theta=THETA, dagger=dagger)
            assert np.linalg.norm(got - want) <= 1e-13 * np.linalg.norm(want)
    finally:
        lq.lattice_destroy(lat)


@pytest.mark.parametrize("theta", [(1, 1, 1, -1), THETA])
def test_both_kernels_store_the_same_bits(lq, theta):
    """One right-hand side of 2048 sites runs on the small kernel, seven of them on the other."""
    dims = (8, 4, 8, 16)
    U = inputs.gauge_field(dims, 0.4, seed=99)
    x = inputs.spinor_field(dims, seed=100, nrhs=7)
    lat = lq.lattice_create(dims)
    try:
        gid = lq.gauge_upload(lat, U)
        dp = lq.dirac_params(0.13, 1.5, theta)
        for dagger in (False, True):
            many = lq.schur_apply(lat, gid, dp, x, precision="fp64", nrhs=7, dagger=dagger)
            one = lq.schur_apply(lat, gid, dp, x[3], precision="fp64", dagger=dagger)
            assert np.array_equal(many[3], one)
    finally:
        lq.lattice_destroy(lat)


@pytest.mark.parametrize("dims", [(2, 2, 2, 2), (6, 2, 6, 4), (8, 8, 10, 14)])
@pytest.mark.parametrize("mu", [0.0, 0.07])
def test_solve_reports_the_true_residual(lq, dims, mu):
    """Three right-hand sides on either kernel (4480 sites are past the rule); the reported residual includes the
    odd sites', which is formed with their solution."""
    U = inputs.gauge_field(dims, 0.3, seed=97)
    b = inputs.spinor_field(dims, seed=98, nrhs=3)
    lat = lq.lattice_create(dims)
    try:
        gid = lq.gauge_upload(lat, U)
        x, info, rc = lq.cg_solve(lat, gid, lq.dirac_params(0.125, 1.3, THETA, mu=mu),
                                  lq.solver_params(tol=1e-12, maxiter=5000, precision="fp64"), b, nrhs=3)
    finally:
        lq.lattice_destroy(lat)
    assert rc == lq.OK, info
    for j in range(3):
        r = b[j] - oracle.dirac_tm(dims, U, 0.125, 1.3, mu, x[j], theta=THETA)
        assert np.linalg.norm(r) <= 1e-12 * np.linalg.norm(b[j])
        assert abs(info[j]["true_resid"] - np.linalg.norm(r) / np.linalg.norm(b[j])) <= 1e-14


@pytest.mark.parametrize("dims", [(4, 4, 4, 4), (8, 12, 10, 26)])
def test_dirac_in_place(lq, dims):
    """D reads the host layout directly; a field that it also writes is copied first."""
    import torch
    U = inputs.gauge_field(dims, 0.4, seed=101)
    psi = torch.from_numpy(inputs.spinor_field(dims, seed=102)).cuda()
    n = psi.numel()
    lat = lq.lattice_create(dims)
    try:
        gid = lq.gauge_upload(lat, U)
        dp = lq.dirac_params(0.13, 1.5)
        want = lq.dirac_apply(lat, gid, dp, psi)
        for shift in (0, 12 * 7):  # the same array, and one that begins seven sites later
            room = torch.zeros(n + shift, dtype=psi.dtype, device="cuda")
            room[:n] = psi.reshape(-1)
            torch.cuda.synchronize()
            got = lq.dirac_apply(lat, gid, dp, room[:n].view(psi.shape), out=room[shift:].view(psi.shape))
            assert torch.equal(got, want)
    finally:
        lq.lattice_destroy(lat)
