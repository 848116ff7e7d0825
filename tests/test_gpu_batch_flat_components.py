"""Each component of the batched form's evaluation on its own, relative to itself, in the
flat systems that planetary ensembles are: no less exact than plain FP64 arithmetic.  A
step of 1e-30 leaves x and v as they are, so the derivatives after it are those of the
initial state with the initial a, a-dot as inputs.

Tolerance, on the median over bodies and systems: 1.5 times the error of the oracle's FP64
evaluation of the same inputs plus one rounding, both against binary128 (the two sum in
different orders).
"""
import numpy as np
import pytest

from paper_2006_02501_gb300 import inputs as I

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
SIZES = [6, 7, 9, 12, 17, 24, 32, 33, 48, 64] * 3


def systems(kind):
    out = []
    for k, n in enumerate(SIZES):
        _, m, x, v, _ = I.planetary_systems(seed=k, S=1, nmin=n, nmax=n)
        if kind in ("thin", "edge"):
            x[:, 2] *= 1e-5
            v[:, 2] *= 1e-5
        if kind == "edge":
            x, v = x[:, [2, 0, 1]], v[:, [2, 0, 1]]
        elif kind == "coplanar":          # one inclined member
            z, w = x[-1, 2], v[-1, 2]
            x[:, 2] = v[:, 2] = 0.0
            x[-1, 2], v[-1, 2] = z, w
        elif kind == "tilted":            # a plane no axis lies along
            R = np.array([[0.6, 0.0, 0.8], [0.0, 1.0, 0.0], [-0.8, 0.0, 0.6]])
            x, v = x @ R, v @ R
        elif kind == "rod":
            x[:, 1:] *= 1e-6
            v[:, 1:] *= 1e-6
        out.append((m, np.ascontiguousarray(x), np.ascontiguousarray(v)))
    return out


@pytest.mark.parametrize("kind", ["plain", "thin", "edge", "coplanar", "tilted", "rod"])
@pytest.mark.parametrize("order", [4, 6, 8])
def test_components(orc, order, kind):
    import paper_2006_02501_gb300 as mh
    p, eps = order // 2 - 1, 1e-3
    parts = systems(kind)
    off = np.concatenate([[0], np.cumsum(SIZES)]).astype(np.int64)
    m, x, v = (np.concatenate([q[k] for q in parts]) for k in range(3))
    with mh.Batch(order, off, m, x, v, np.full(len(SIZES), 1e-30), eps) as b:
        d0 = b.sync()[3].copy()
        b.step(1, 1)
        d = b.sync()[3]
    K = min(p + 1, 2 * p)
    errs = {"gpu": [], "fp64": []}
    for a, z in zip(off, off[1:]):
        tr = np.stack([x[a:z], v[a:z]] + [d0[a:z, k] for k in range(p - 1)], 1)
        ref = orc.dd_evaluate(m[a:z], np.stack([tr, np.zeros_like(tr)], -1), eps)
        for name, got in (("gpu", d[a:z, :K]), ("fp64", orc.evaluate(m[a:z], tr, eps)[:, :K])):
            hi = ref[1:, :K, :, 0]
            with np.errstate(divide="ignore", invalid="ignore"):
                errs[name].append(np.abs((got[1:] - hi) - ref[1:, :K, :, 1]) / np.abs(hi))
    gpu, fp64 = (np.nanmedian(np.concatenate(errs[k]), axis=0) for k in ("gpu", "fp64"))
    assert np.all(gpu <= 1.5 * fp64 + 2.0 ** -53), (gpu, fp64)
