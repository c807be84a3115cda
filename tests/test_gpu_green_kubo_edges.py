"""Green-Kubo sums at the edges of their kernels: lags either side of the scan's 256-lag chunks, one
trajectory to many, series shorter than a block, the largest lag.

Tolerance 1e-13 acf(0) and 1e-13 of the integral with acf(0) for every lag: sums of up to 5 x 9 x 700 products in FP64 in another order,
about sqrt(n) 2^-53 of the sum of magnitudes, which acf(0) bounds."""
import numpy as np
import pytest

from oracle import green_kubo

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n_traj,n_steps,max_lag", [(1, 2, 1), (1, 300, 255), (7, 300, 256), (8, 700, 511), (9, 700, 512),
                                                    (17, 520, 519)])
def test_chunk_edges(n_traj, n_steps, max_lag):
    from paper_2006_03697_gb300 import build
    build.build()
    from paper_2006_03697_gb300 import sq
    rng = np.random.Generator(np.random.PCG64(n_traj * 1000 + n_steps))
    sig = 0.01 * rng.normal(size=(n_traj, n_steps, 3, 3))
    dt, vol, kT = 10.0, 500.0, 3.0
    eta_ref, acf_ref = green_kubo.viscosity(sig, dt, vol, kT, max_lag)
    eta, acf = sq.sq_green_kubo(sig, dt, vol, kT, max_lag)
    np.testing.assert_allclose(acf, acf_ref, rtol=0.0, atol=1e-13 * acf_ref[0])
    scale = vol / kT * dt * (max_lag + 1) * acf_ref[0]
    np.testing.assert_allclose(eta, eta_ref, rtol=0.0, atol=1e-13 * scale)
