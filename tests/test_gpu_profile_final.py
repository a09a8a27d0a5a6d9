"""Byte counts of the kernels that close a solve.

Three right-hand sides of an FP64 solve reach the target by their recursion, in
whatever polls: the correction and the update of x are charged once for each of
them (and the site blocks once a launch), and the odd solution for its two site
blocks, inverse and A.
"""
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


def test_bytes(lq):
    dims, nrhs, vh, spinor, blocks = (4, 4, 4, 8), 3, 256, 192.0, 576.0
    b = inputs.spinor_field(dims, seed=702, nrhs=nrhs)
    lat = lq.lattice_create(dims)
    try:
        gid = lq.gauge_upload(lat, inputs.gauge_field(dims, 0.3, seed=701))
        args = (lat, gid, lq.dirac_params(0.12, 1.2), lq.solver_params(tol=1e-10, precision="fp64"), b)
        lq.cg_solve(*args, nrhs=nrhs)  # autotunes
        lq.profile_reset()
        _, info, rc = lq.cg_solve(*args, nrhs=nrhs)
        prof = lq.profile_read()
    finally:
        lq.lattice_destroy(lat)
    assert rc == lq.OK and [i["iters_outer"] for i in info] == [1] * nrhs
    assert prof["cg_x_update"]["bytes"] == vh * nrhs * 4 * spinor  # e and x, read and written
    site = prof["cg_e_site"]
    assert site["bytes"] == vh * (nrhs * 3 * spinor + site["launches"] * blocks)  # e in and out, p
    assert prof["hop_f64_clovsum"]["bytes"] == vh * (nrhs * 3 * spinor + 8 * 144.0 + 2 * blocks)
