"""A softening whose cube leaves the range of doubles gives zero accelerations, as in FP64."""
import numpy as np
import pytest

from helpers import kepler_traj
from paper_2006_02501_gb300 import inputs as I

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.mark.parametrize("eps", [1e70, 1e110, 1e150])
def test_pair_eval(orc, eps):
    import paper_2006_02501_gb300 as mh
    N = 1100
    m, x, v = I.smbh_disc(seed=3, N=N - 1)
    tr = kepler_traj(m, x, v, 3) * 1e25
    rows = torch.from_numpy(np.ascontiguousarray(tr.reshape(N, -1).T)).cuda()
    out = torch.empty((12, N), dtype=torch.float64, device="cuda")
    mh.pair_eval(3, mh.MH_PREC_FP64, torch.from_numpy(m).cuda(), rows, eps, out)
    got = out.cpu().numpy().T.reshape(N, 4, 3)
    ref = orc.evaluate(m, tr, eps)
    assert np.abs(got - ref).max() <= 1e-13 * np.abs(ref).max()


@pytest.mark.parametrize("eps", [1e110, 1e150])
def test_symmetric(eps):
    import paper_2006_02501_gb300 as mh
    m, x, v = I.smbh_disc(seed=3, N=299)
    with mh.Simulation(6, m, x, v, eps, symmetric=2) as sim:
        assert np.all(sim.sync()[3] == 0.0)
