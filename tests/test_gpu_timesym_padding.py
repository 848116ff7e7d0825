"""Eq. 24's maximum must come from pairs of bodies only: the pair-symmetric kernels pad
the last block with massless positions, just outside the system's largest coordinate
(orders up to 8) or at 1e6 (above), and a body beside them must not shorten the step.

Tolerance: that of test_timesym_pair_symmetric_kernel (the step sizes agree to rounding).
"""
import numpy as np
import pytest

from paper_2006_02501_gb300 import inputs as I

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.mark.parametrize("order,n,place", [(4, 300, 1 - 1e-3), (6, 130, 1 - 1e-3), (8, 300, 1 - 1e-3),
                                           (8, 255, 1 - 1e-6), (8, 256, 1 - 1e-3), (10, 300, 1e6 + 0.25)])
def test_body_beside_the_padding(orc, order, n, place):
    import paper_2006_02501_gb300 as mh
    m, x, v = I.disc_100(seed=4, n=n - 1, m=1e-8, a_lo=0.1, a_hi=0.7)
    k = n // 2
    m[k], x[k], v[k] = 1e-3, [0.999, 0.0, 0.0], [0.0, 1.0, 0.0]
    assert np.abs(x).max() < 1.0
    scale = place / 0.999
    x, v = x * scale, v * scale ** -0.5
    x[k, 0] = place
    eta, n_iter, K = 0.02, 3, 4
    with mh.Simulation(order, m, x, v, 0.0, timesym_eta=eta, symmetric=2) as sim:
        sim.step_timesym(K, n_iter)
        t, xg, _, _ = sim.sync()
    ref = orc.State(order, m, x, v, 0.0)
    ref.step_timesym(eta, n_iter, K)
    assert abs(t - ref.t) / ref.t < 1e-12
    assert np.abs(xg - ref.x).max() < 1e-12 * scale
