"""The exponential of the link update for large exponents with a double eigenvalue.

An HMC trajectory of one step at beta = 1e-30 (no force to speak of) gives U' = exp(eps P) U.
P = i c Q diag(1, 1, -2) Q^dag / sqrt(6) has |P|_F = c and exp(eps P) is known.
Rounding of P and each of the log2(2 eps c) squarings cost a few 2^-53 of
the exponent: bound 40 (1 + eps c) 2^-53, where squaring only the coefficients of
the Cayley-Hamilton form loses (eps c)^2 2^-53.
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


@pytest.mark.parametrize("size", [0.3, 5.0, 30.0, 1000.0, 4000.0])
def test_double_eigenvalue(lq, size):
    dims, c = (4, 4, 4, 4), 2.0
    n = 4 * 256
    rng = np.random.default_rng(7)
    Q = np.linalg.qr(rng.normal(size=(n, 3, 3)) + 1j * rng.normal(size=(n, 3, 3)))[0]
    d = np.array([1.0, 1.0, -2.0]) * c / np.sqrt(6.0)
    H = (Q * d) @ Q.conj().transpose(0, 2, 1)
    mom = np.einsum("aij,nji->na", inputs.gell_mann(), H).real  # P = sum_a mom_a i lambda_a / 2
    E = (Q * np.exp(1j * size / c * d)) @ Q.conj().transpose(0, 2, 1)
    U = inputs.gauge_field(dims, 0.4, seed=601)
    lat = lq.lattice_create(dims)
    try:
        gid = lq.gauge_upload(lat, U)
        acc, _ = lq.hmc_trajectory(lat, gid, 1e-30, size / c, 1, mom.reshape(4, 4, 4, 4, 4, 8), 1e-300)
        assert acc
        got = lq.gauge_download(lat, gid, dims)
    finally:
        lq.lattice_destroy(lat)
    want = E.reshape(U.shape) @ U
    assert np.max(np.abs(got - want)) <= 40 * (1 + size) * 2.0 ** -53
