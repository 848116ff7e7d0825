"""A body whose state has become NaN (reported by the next synchronisation) does not keep
the other bodies' step from converging."""
import numpy as np
import pytest

from paper_2006_02501_gb300 import inputs as I

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.mark.parametrize("order", [4, 8])
def test_passes_with_coinciding_bodies(order):
    import paper_2006_02501_gb300 as mh
    m, x, v = I.disc_100(seed=2)
    with mh.Simulation(order, m, x, v, 0.0) as sim:
        plain = sim.step_converge(1e-3, 1e-12, 30)
    assert plain < 15
    x[41], v[41] = x[40], v[40]
    m[40] = m[41] = 0.0                      # the others do not feel them
    with mh.Simulation(order, m, x, v, 0.0) as sim:
        assert sim.step_converge(1e-3, 1e-12, 30) <= plain
        with pytest.raises(mh.MHError):
            sim.sync()
