"""GPU solves where the site block of an even site is singular or nearly so.

D is invertible all the same: only the odd sites' blocks have to be.  kappa
c_sw is set to (1 - delta) / lambda, with lambda the largest eigenvalue of the
clover term, which the chosen field has on an even site, 1.26 times the odd
sites' largest: that block then has the eigenvalue delta.  From a small delta
down to 0 (an inverse of infinities), and on both sides of the line up to which
the solver divides the even site term out (entries of 8: delta 0.0345).
Iterations: Dhat needs 130 to 390 here, so 600 is a stall.
"""
import numpy as np
import pytest

import oracle
from paper_2503_16994_gb300 import inputs

pytestmark = pytest.mark.gpu
DIMS, KAPPA = (4, 4, 4, 6), 0.06


@pytest.fixture(scope="module")
def lq():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__
    __graft_entry__.build()
    from paper_2503_16994_gb300 import lqcd
    return lqcd


@pytest.fixture(scope="module")
def field():
    """(links, lambda): the blocks are A_s = 1 - kappa c_sw K_s, K from the oracle's field strength."""
    U = inputs.gauge_field(DIMS, 0.4, seed=8)
    xy, xz, xt, yz, yt, zt = (oracle.field_strength(DIMS, U)[..., q, :, :] for q in range(6))
    lam = 0.0
    for sg in (1, -1):
        mx, my, mz = yz + sg * xt, -xz + sg * yt, xy + sg * zt
        K = np.zeros(mx.shape[:-2] + (6, 6), complex)
        K[..., :3, :3], K[..., 3:, 3:] = 1j * mz, -1j * mz
        K[..., :3, 3:], K[..., 3:, :3] = 1j * (mx - 1j * my), 1j * (mx + 1j * my)
        lam = np.maximum(lam, np.linalg.eigvalsh(K)[..., -1])
    t, z, y, x = np.indices(DIMS[::-1])
    even = (x + y + z + t) % 2 == 0
    assert lam[even].max() > 1.2 * lam[~even].max()
    return U, lam[even].max()


@pytest.mark.parametrize("prec", ["fp64", "fp32", "fp16"])
@pytest.mark.parametrize("delta", [0.045, 0.03, 1e-4, 1e-7, 0.0])
@pytest.mark.parametrize("mu", [0.0, 1e-7])
def test_solve(lq, field, prec, delta, mu):
    U, lam = field
    nrhs, tol, csw = 2, 1e-10, (1 - delta) / field[1] / KAPPA
    b = inputs.spinor_field(DIMS, seed=9, nrhs=nrhs)
    lat = lq.lattice_create(DIMS)
    try:
        gid = lq.gauge_upload(lat, U)
        x, info, rc = lq.cg_solve(lat, gid, lq.dirac_params(KAPPA, csw, mu=mu),
                                  lq.solver_params(tol=tol, maxiter=600, precision=prec), b, nrhs=nrhs)
    finally:
        lq.lattice_destroy(lat)
    assert rc == lq.OK, info
    for j in range(nrhs):
        r = b[j] - oracle.dirac_tm(DIMS, U, KAPPA, csw, mu, x[j])
        assert np.linalg.norm(r) <= 1.001 * tol * np.linalg.norm(b[j])


def test_batched_and_served(lq, field):
    U, lam = field
    dp = lq.dirac_params(KAPPA, (1 - 1e-7) / lam / KAPPA)
    sp = lq.solver_params(tol=1e-9, maxiter=600, precision="fp16")
    ref, *_ = oracle.pion(DIMS, U, KAPPA, (1 - 1e-7) / lam / KAPPA, (1, 0, 2, 3), tol=1e-12)
    lat = lq.lattice_create(DIMS)
    srv = lq.serve_create(max_slots=2)
    try:
        gid = lq.gauge_upload(lat, U)
        corrs, _, _, rc = lq.pion_corr_batch([(lat, gid, dp, (1, 0, 2, 3), DIMS[3])] * 2, sp)
        assert rc == lq.OK
        ticket = lq.serve_submit(srv, lq.serve_gauge(srv, DIMS, U), dp, sp, (1, 0, 2, 3))
        rc, corr, _, _ = lq.serve_poll(srv, ticket, DIMS[3], timeout_ms=60000)
        assert rc == lq.OK
    finally:
        lq.serve_destroy(srv)
        lq.lattice_destroy(lat)
    for c in corrs + [corr]:
        assert np.all(np.abs(c - ref) <= 1e-6 * np.abs(ref))
