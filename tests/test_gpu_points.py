"""Point kernels at the edges of their CTAs and for every instantiation:
degrees 1..3, scalar and 3-vector, FP32, FP16 and BF16 blocks, against the
FP64 oracle.  Degree 4 and unequal degrees keep the loops over any degree.

Values are held to 1e-5 max|c| (FP32) plus the storage's 1.02 s u with s <=
max|c| (u = 2^-11 or 2^-8; point evaluation rounds nothing else).  The
gradient of an axis sums (p + 1)^3 terms of size p * iw * max|c| twice over,
so its bars are those times 2 p iw (iw = 1 / the element's side).
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from oracle.oracle import Oracle
from paper_1707_01170_gb300 import lrvol as lv
from paper_1707_01170_gb300.synth import volumes as V
from paper_1707_01170_gb300.synth.lrgen import Stream

pytestmark = pytest.mark.gpu
U = {lv.STORE_F32: 0.0, lv.STORE_F16: 2.0 ** -11, lv.STORE_BF16: 2.0 ** -8}


def _points(n, seed):
    """Inside, on faces and corners, and outside."""
    X = Stream(seed, 3 * n + 8).take(3 * n).reshape(n, 3).astype(np.float32)
    k = np.arange(n)
    X[k % 7 == 1] = np.round(X[k % 7 == 1] * 4) / 4
    X[k % 11 == 2, 0] = 1.0
    X[k % 13 == 3] = (k[k % 13 == 3, None] // 13 + np.arange(3)) % 2
    X[k % 17 == 5, 1] = 1.0 + 2.0 ** -23
    X[k % 19 == 6, 2] = -1e-7
    X[k % 23 == 7, 0] = np.nan
    return X


@pytest.mark.parametrize("ncomp", [1, 3])
@pytest.mark.parametrize("deg", [(1, 1, 1), (2, 2, 2), (3, 3, 3), (4, 4, 4), (1, 2, 3), (3, 3, 2)])
def test_values_and_gradients(deg, ncomp):
    vol = V.refined_ball(deg, (3, 3, 3), centres=((0.4, 0.55, 0.5),), radii=(0.35,), ncomp=ncomp, seed=7)
    orc, cmax = Oracle(vol), float(np.abs(vol.coef).max())
    X = _points(641, 40 + sum(deg))
    inside = np.all((X >= 0) & (X <= 1), axis=1)
    val, elem = orc.eval(X[inside], return_elem=True)
    for storage, u in U.items():
        gv = lv.Volume(vol).build_accel((4, 4, 4)).to_bezier(storage)
        bar = cmax * (1e-5 + 1.02 * u)
        for n in (0, 1, 127, 128, 129, 641):
            got = gv.eval(torch.from_numpy(X[:n].copy()).cuda().reshape(n, 3)).cpu().numpy().astype(np.float64)
            keep = inside[:n]
            assert got.shape == (n, ncomp) and np.all(got[~keep] == 0.0)
            assert np.all(np.abs(got[keep] - val[:keep.sum()]) <= bar)
        if ncomp == 1:
            want_v, want_g = orc.eval_grad(X[inside])
            got = gv.eval_grad(torch.from_numpy(X).cuda()).cpu().numpy().astype(np.float64)
            assert np.all(got[~inside] == 0.0)
            box = vol.elem_box[elem]
            gbar = 2 * max(deg) / (box[:, 3:] - box[:, :3]) * bar
            assert np.all(np.abs(got[inside, 0] - want_v.reshape(-1)) <= bar)
            assert np.all(np.abs(got[inside, 1:] - want_g[:, 0]) <= gbar)
        gv.close()
