"""Each component of a .. a^(3) on its own, relative to itself: the fixed-point evaluation
must keep a small component (a disc's vertical one) as exactly as FP64 arithmetic does,
where the bulk of the system is flat and one body is not as well as where all are.

Tolerance, on the median over bodies: the 40 to 80 FP64 sums of 32 terms each round to
2^-53 / sqrt(12) of the sum, 2e-16 .. 3e-16 in all; a term of a^(3) has parts up to 6
times its size: 1.8e-15, eight units of 2^-52.  Against binary128.
"""
import numpy as np
import pytest

from paper_2006_02501_gb300 import inputs as I

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
TOL = 8 * 2.0 ** -52
KINDS = ["disc", "thin", "inclined", "coplanar", "sheet", "edge", "cluster", "sorted", "rod"]


def system(kind, N):
    g = np.random.default_rng(N)
    if kind in ("cluster", "sorted", "rod"):
        m, x, v = np.full(N, 1.0 / N), g.normal(size=(N, 3)), g.normal(size=(N, 3))
        if kind == "sorted":
            k = np.argsort(x[:, 2])
            x, v = x[k], v[k]
        if kind == "rod":
            x[:, 1:] *= 1e-6
            v[:, 1:] *= 1e-6
        return m, x, v
    m, x, v = I.smbh_disc(seed=N, N=N - 1, sigma_i=0.025 if kind == "disc" else 1e-6)
    if kind in ("inclined", "coplanar"):
        k = N // 3
        if kind == "coplanar":
            x[:, 2] = v[:, 2] = 0.0
        m[k] = 0.0 if kind == "inclined" else 1e-6
        x[k], v[k] = [0.3, 0.2, 0.4], [0.5, -0.7, 0.6]
    elif kind == "sheet":
        x[:, 2] += 5.0
        v[:, 2] += 0.7
    elif kind == "edge":
        x, v = x[:, [2, 0, 1]], v[:, [2, 0, 1]]
    return m, np.ascontiguousarray(x), np.ascontiguousarray(v)


def medians(got, ref2):
    """Median over bodies of each component's relative error, (P+1, 3)."""
    ref = ref2[..., 0]
    e = np.abs((got - ref) - ref2[..., 1])
    assert np.all(got[ref == 0.0] == 0.0)
    return np.array([[np.median(e[:, k, c][ref[:, k, c] != 0] / np.abs(ref[:, k, c][ref[:, k, c] != 0]))
                      if np.any(ref[:, k, c]) else 0.0 for c in range(3)] for k in range(ref.shape[1])])


def pairs(a):
    return np.stack([a, np.zeros_like(a)], -1)


@pytest.mark.parametrize("kind", KINDS)
@pytest.mark.parametrize("P", [1, 2, 3])
def test_ordered(orc, kind, P):
    import paper_2006_02501_gb300 as mh
    N, n = 1300, 160
    m, x, v = system(kind, N)
    d = orc.initialise(6, m, x, v, 1e-4)
    tr = np.stack([x, v, d[:, 0], d[:, 1]][:P + 1], 1)
    rows = torch.from_numpy(np.ascontiguousarray(tr.reshape(N, -1).T)).cuda()
    out = torch.empty((3 * (P + 1), N), dtype=torch.float64, device="cuda")
    mh.pair_eval(P, mh.MH_PREC_FP64, torch.from_numpy(m).cuda(), rows, 1e-4, out)
    got = out.cpu().numpy().T.reshape(N, P + 1, 3)[1:n]
    assert medians(got, orc.dd_evaluate(m, pairs(tr), 1e-4, i0=1, i1=n)).max() < TOL


@pytest.mark.parametrize("kind", KINDS)
def test_symmetric(orc, kind):
    """The initialisation passes P = 1 (a, a-dot) and P = 3 (a'', a''')."""
    import paper_2006_02501_gb300 as mh
    N, n = 1300, 160
    m, x, v = system(kind, N)
    with mh.Simulation(6, m, x, v, 1e-4, symmetric=2) as sim:
        d = sim.sync()[3]
    tr = np.stack([x, v, d[:, 0], d[:, 1]], 1)
    assert medians(d[1:n], orc.dd_evaluate(m, pairs(tr), 1e-4, i0=1, i1=n)).max() < TOL
