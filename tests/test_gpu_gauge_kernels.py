"""GPU force, exponential and Laplacian of the flows at the sizes where they can go wrong.

Extents of 2 (both neighbours are one site, and every staple slot is written
by a wrapped hop), lattices that do not fill a block, step sizes whose stage
exponents need squarings, and the force without scratch (the staples formed
per link), which must give the same links.  Bounds: a stage is a few hundred
FP64 roundings (1e-16 each) and the flow amplifies them by less than 100 over
these steps, so 1e-12 on O(1) links.
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


@pytest.mark.parametrize("dims", [(2, 2, 2, 2), (2, 4, 6, 2), (6, 2, 4, 10)])
@pytest.mark.parametrize("eps,n", [(0.02, 3), (0.3, 1)])
def test_fermion_flow_edges(lq, dims, eps, n):
    U = inputs.gauge_field(dims, 0.4, seed=91)
    psi = inputs.spinor_field(dims, seed=92, nrhs=3)
    theta = (np.exp(0.3j), 1, np.exp(-0.7j), -1)
    lat = lq.lattice_create(dims)
    try:
        gid = lq.gauge_upload(lat, U)
        got = lq.fermion_flow(lat, gid, lq.dirac_params(0.13, 0.0, theta), psi, eps, n, nrhs=3)
        Uf = lq.gauge_download(lat, gid, dims)
    finally:
        lq.lattice_destroy(lat)
    Uo, want = oracle.fermion_flow(dims, U, psi, eps, n, theta=theta, nrhs=3)
    assert np.max(np.abs(Uf - Uo)) <= 1e-12
    assert np.linalg.norm(got - want) <= 1e-12 * np.linalg.norm(want)


def test_flow_without_scratch(lq):
    """16^4 needs 38 MB for the accumulator and 142 MB of scratch: with 100 MB free only the first fits."""
    import torch
    dims = (16, 16, 16, 16)
    U = inputs.gauge_field(dims, 0.4, seed=93)
    lat = lq.lattice_create(dims)
    hog = None
    try:
        gid = [lq.gauge_upload(lat, U), lq.gauge_upload(lat, U)]
        lq.gauge_flow(lat, gid[0], 0.02, 2)
        torch.cuda.synchronize()
        free, _ = torch.cuda.mem_get_info()
        hog = torch.empty(free - (100 << 20), dtype=torch.uint8, device="cuda")
        lq.gauge_flow(lat, gid[1], 0.02, 2)
        hog = None
        torch.cuda.empty_cache()
        a, b = (lq.gauge_download(lat, g, dims) for g in gid)
    finally:
        del hog
        lq.lattice_destroy(lat)
    assert np.max(np.abs(a - b)) <= 1e-13
    assert np.max(np.abs(a - U)) > 1e-3
