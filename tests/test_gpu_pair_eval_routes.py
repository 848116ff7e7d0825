"""mh_pair_eval at both sides of the sizes where its evaluation changes between FP64 and
fixed point (fix_pays), with the many partial-sum slots that small calls are split into.

Tolerance: that of test_gpu_fixed_point (1e-13 of the largest component per body and order).
"""
import numpy as np
import pytest

from helpers import kepler_traj
from paper_2006_02501_gb300 import inputs as I

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.mark.parametrize("P,N,ni", [(1, 799, 799), (1, 800, 800), (2, 759, 759), (2, 760, 760), (3, 724, 724),
                                    (3, 725, 725), (3, 16384, 64), (3, 16384, 65), (3, 16385, 64), (2, 16385, 36),
                                    (1, 8192, 79), (3, 5, 3), (4, 700, 699), (3, 1025, 1)])
def test_both_sides(orc, P, N, ni):
    import paper_2006_02501_gb300 as mh
    m, x, v = I.smbh_disc(seed=N, N=N - 1)
    tr = np.zeros((N, P + 1, 3))
    tr[:, :min(P, 3) + 1] = kepler_traj(m, x, v, min(P, 3))
    rows = torch.from_numpy(np.ascontiguousarray(tr.reshape(N, -1).T)).cuda()
    out = torch.empty((3 * (P + 1), ni), dtype=torch.float64, device="cuda")
    i0 = N - ni
    mh.pair_eval(P, mh.MH_PREC_FP64, torch.from_numpy(m).cuda(), rows, 1e-4, out, i0=i0, i1=N)
    got = out.cpu().numpy().T.reshape(ni, P + 1, 3)
    ref = orc.evaluate(m, tr, 1e-4, i0=i0, i1=N)
    scale = np.abs(ref).max(-1)
    assert (np.abs(got - ref).max(-1) / np.where(scale > 0, scale, 1.0)).max() < 1e-13
