"""The flows give the same bits whether or not the device has room for the force's scratch,
and the scratch leaves as much memory free as it takes.

Each call runs with plenty of memory and again with so little that its other
fields fit and the scratch (2160 bytes a site) does not; the profile shows
which force ran.  Gauge flow, HMC, fermion flow and backflow.
"""
import numpy as np
import pytest

from paper_2503_16994_gb300 import inputs

pytestmark = pytest.mark.gpu
MB = 1 << 20


@pytest.fixture(scope="module")
def lq():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__
    __graft_entry__.build()
    from paper_2503_16994_gb300 import lqcd
    return lqcd


def call(lq, kind, lat, gid, dims, psi, mom):
    """(outputs, names of the profiled kernels); psi: a fresh copy on the device"""
    p = lq.dirac_params(0.12, 0.0)
    lq.profile_reset()
    if kind == "flow":
        lq.gauge_flow(lat, gid, 0.02, 2)
    elif kind == "hmc":
        acc, dH = lq.hmc_trajectory(lat, gid, 5.8, 0.05, 2, mom, 1e-9)
        assert acc
        return [dH, lq.gauge_download(lat, gid, dims)], set(lq.profile_read())
    elif kind == "fermion":
        lq.fermion_flow(lat, gid, p, psi, 0.02, 2)
    else:
        lq.fermion_backflow(lat, gid, p, psi, 0.02, 2, nsave=2)
    names = set(lq.profile_read())
    return [psi.cpu().numpy(), lq.gauge_download(lat, gid, dims)], names


# megabytes left free: the call's other fields take 38 (flow), 80 (hmc), 76 (fermion) and 252 (backflow) on 16^4,
# the links read back 38 more, the scratch's first part 113
@pytest.mark.parametrize("kind,left", [("flow", 100), ("hmc", 150), ("fermion", 140), ("back", 320)])
def test_same_bits(lq, kind, left):
    import torch
    dims = (16, 16, 16, 16)
    U = inputs.gauge_field(dims, 0.4, seed=93)
    psi0 = torch.from_numpy(inputs.spinor_field(dims, seed=94)).cuda()
    mom = inputs.normals(95, 0, 16 ** 4 * 32).reshape(dims + (4, 8))
    lat = lq.lattice_create(dims)
    hog, got, names = None, [], []
    try:
        ids = [lq.gauge_upload(lat, U), lq.gauge_upload(lat, U)]
        psis = [psi0.clone(), psi0.clone()]
        for k in range(2):
            if k == 1:
                torch.cuda.synchronize()
                free, _ = torch.cuda.mem_get_info()
                hog = torch.empty(free - left * MB, dtype=torch.uint8, device="cuda")
            out, used = call(lq, kind, lat, ids[k], dims, psis[k], mom)
            got.append(out)
            names.append(used)
    finally:
        del hog
        torch.cuda.empty_cache()
        lq.lattice_destroy(lat)
    for a, b in zip(*got):
        assert np.array_equal(a, b)
    assert "force_no_scratch" not in names[0] and "force_no_scratch" in names[1]
    assert np.max(np.abs(got[0][1] - U)) > 1e-3 or kind == "back"


@pytest.mark.parametrize("left,scratch", [(300, False), (360, True)])
def test_scratch_leaves_as_much_as_it_takes(lq, left, scratch):
    """16^4: 38 MB for the accumulator, 142 of scratch: 262 and 322 MB are free when it is decided."""
    import torch
    dims = (16, 16, 16, 16)
    lat = lq.lattice_create(dims)
    hog = None
    try:
        gid = lq.gauge_upload(lat, inputs.gauge_field(dims, 0.4, seed=93))
        torch.cuda.synchronize()
        free, _ = torch.cuda.mem_get_info()
        hog = torch.empty(free - left * MB, dtype=torch.uint8, device="cuda")
        lq.profile_reset()
        lq.gauge_flow(lat, gid, 0.02, 1)
        names = set(lq.profile_read())
    finally:
        del hog
        torch.cuda.empty_cache()
        lq.lattice_destroy(lat)
    assert ("force_no_scratch" not in names) == scratch
