"""Batched propagators whose jobs share a gauge field and its site terms.

The first job that needs a clover field (or the links of SF boundaries) builds
it on its own stream; the others have to wait for it.  On fields uploaded anew
each time, with sources, masses and boundaries mixed, the batch gives the
correlators of one call per job.  Both stop at 1e-10, so C(t) agrees to a few
1e-10 of its largest value.
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


@pytest.mark.parametrize("bc", ["periodic", "sf"])
def test_jobs_on_one_gauge_field(lq, bc):
    dims = (16, 16, 8, 16)
    sp = lq.solver_params(tol=1e-10, precision="fp32")
    work = [(0.12, (0, 1, 2, 3)), (0.12, (5, 4, 3, 9)), (0.118, (1, 1, 1, 1)), (0.12, (2, 0, 2, 4))]
    lat = lq.lattice_create(dims)
    try:
        for seed in range(4):
            U = inputs.gauge_field(dims, 0.3, seed=500 + seed)
            gid = lq.gauge_upload(lat, U)
            dps = [lq.dirac_params(k, 1.2, bc=bc) for k, _ in work]
            got, _, _, rc = lq.pion_corr_batch([(lat, gid, dp, src, dims[3]) for dp, (_, src) in zip(dps, work)], sp)
            assert rc == lq.OK
            for c, dp, (_, src) in zip(got, dps, work):
                ref, _, _, rc = lq.pion_corr(lat, gid, dp, sp, src, dims=dims)
                assert rc == lq.OK
                assert np.max(np.abs(c - ref)) <= 1e-8 * np.max(ref)
            lq.gauge_free(lat, gid)
    finally:
        lq.lattice_destroy(lat)
