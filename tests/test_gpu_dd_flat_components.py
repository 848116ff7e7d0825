"""Each component of a .. a^(3) on its own, relative to itself, in the double-double form:
its integer arithmetic must keep a small component as exactly as double-double does, where
the bulk of a system is flat and one body is not as well as where all are.

Tolerance, on the median over bodies: 2^-102, the double-double kernels' own size (a
product or sum to 2^-104 .. 2^-105 and a^(3)'s parts up to 4 times its size).
"""
import numpy as np
import pytest

from test_gpu_flat_components import KINDS, system

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
TOL = 2.0 ** -102
# (not "sheet": an offset of 5e6 times the thickness leaves binary128, the reference, 1e-31 .. 4e-31)
DD_KINDS = [k for k in KINDS if k != "sheet"]


def with_low_words(a, seed):
    lo = a * np.random.default_rng(seed).uniform(-1e-16, 1e-16, a.shape)
    hi = a + lo
    return np.stack([hi, (a - hi) + lo], -1)


def medians(got2, ref2):
    ref = ref2[..., 0]
    e = np.abs((got2[..., 0] - ref) + (got2[..., 1] - ref2[..., 1]))
    assert np.all(got2[..., 0][ref == 0.0] == 0.0)
    return np.array([[np.median(e[:, k, c][ref[:, k, c] != 0] / np.abs(ref[:, k, c][ref[:, k, c] != 0]))
                      if np.any(ref[:, k, c]) else 0.0 for c in range(3)] for k in range(ref.shape[1])])


@pytest.mark.parametrize("symmetric", [0, 2])
@pytest.mark.parametrize("kind", DD_KINDS)
@pytest.mark.parametrize("P,N", [(1, 200), (2, 200), (3, 300)])
def test_evaluation(orc, kind, P, N, symmetric):
    import paper_2006_02501_gb300 as mh
    m, x, v = system(kind, N)
    d = orc.initialise(6, m, x, v, 1e-4)
    tr2 = with_low_words(np.stack([x, v, d[:, 0], d[:, 1]][:P + 1], 1), N)
    got = mh.dd_pair_eval(P, m, tr2, 1e-4, symmetric=symmetric)
    assert medians(got[1:], orc.dd_evaluate(m, tr2, 1e-4)[1:]).max() < TOL


@pytest.mark.parametrize("kind", DD_KINDS)
def test_batch(orc, kind):
    """The initialisation passes P = 1 (a, a-dot) and P = 3 (a'', a''') of systems of 8 to 64 bodies."""
    import paper_2006_02501_gb300 as mh
    sizes = [64, 48, 33, 32, 17, 8] * 3
    parts = [system(kind, n) for n in sizes]
    off = np.concatenate([[0], np.cumsum(sizes)])
    m, x, v = (np.concatenate([q[k] for q in parts]) for k in range(3))
    with mh.DDBatch(6, off, m, x, v, np.full(len(sizes), 1e-4), 1e-4) as b:
        d = b.sync()[3]
    got, ref = [], []
    for a, z in zip(off, off[1:]):
        xv = np.stack([x[a:z], v[a:z]], 1)
        tr2 = np.concatenate([np.stack([xv, np.zeros_like(xv)], -1), d[a:z, :2]], 1)
        got.append(d[a + 1:z])
        ref.append(orc.dd_evaluate(m[a:z], tr2, 1e-4)[1:])
    assert medians(np.concatenate(got), np.concatenate(ref)).max() < TOL
