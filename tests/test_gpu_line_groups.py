"""Lines by four lanes against lines by one lane: the same seeds in a rake small
enough for groups of lanes and repeated in one too large for them give the same
bits, for every degree, storage and method, in forests with and without trees, with
lines that leave the cube, meet the cap, end at t_end, start outside, and run into a
field that is not finite.
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_1707_01170_gb300 import lrvol as lv
from paper_1707_01170_gb300.synth import volumes as V
from paper_1707_01170_gb300.synth.lrgen import Stream

pytestmark = pytest.mark.gpu


def _seeds(n):
    x = Stream(91, 3 * n + 8).take(3 * n).reshape(n, 3)
    x[0], x[1], x[2], x[3] = (1.0, 1.0, 1.0), (0.0, 0.5, 1.0), (1.25, 0.5, 0.5), (0.5, np.nan, 0.5)
    return x


def _trace(gv, seeds, method, rule, h, tol):
    n = len(seeds)
    out = (torch.zeros((n, 96, 4), dtype=torch.float64, device="cuda"),
           torch.zeros(n, dtype=torch.int32, device="cuda"), torch.zeros(n, dtype=torch.int32, device="cuda"))
    lv.streamlines(gv, seeds, method, rule, h, 0.75, tol=tol, max_samples=96, out=out)
    return [t.cpu() for t in out]


@pytest.mark.parametrize("storage", [lv.STORE_F32, lv.STORE_F16, lv.STORE_BF16])
@pytest.mark.parametrize("deg", [1, 2, 3])
@pytest.mark.parametrize("finite", [True, False])
@pytest.mark.parametrize("side,blocks", [(3, 4), (4, 8)])     # a forest with trees, and one without
def test_groups_equal_single_lanes(deg, storage, finite, side, blocks):
    vol = V.refined_ball((deg,) * 3, (side,) * 3, radii=(0.35,), ncomp=3, seed=6)
    vol.coef = 2 * vol.coef - 1
    if not finite:
        vol.coef[len(vol.coef) // 2] = (np.inf, np.nan, 1.0)
    gv = lv.Volume(vol).build_accel((blocks,) * 3).to_bezier(storage)
    assert (gv.stats()["n_nodes"] > 0) == (side == 3)
    few, reps = _seeds(37), 2400             # 88,800 lines: a lane each, every lane of a warp in use
    small = torch.from_numpy(few).cuda()
    large = small.repeat(reps, 1)
    seen = set()
    for method, rule, h, tol in (("RK1", "fixed", 0.01, 0.0), ("RK4", "heuristic", 1.0, 0.0), ("RKF5", "heuristic", 2.0, 0.0),
                                 ("HE", "adaptive", 0.0, 1e-5), ("RKF45", "adaptive", 0.3, 1e-7)):
        a, b = _trace(gv, small, method, rule, h, tol), _trace(gv, large, method, rule, h, tol)
        for x, y in zip(a, b):
            x, y = x.numpy(), y.numpy().reshape(reps, *x.shape)
            assert np.array_equal(x.view(np.int64 if x.dtype == np.float64 else np.int32),
                                  y[0].view(np.int64 if x.dtype == np.float64 else np.int32))
            assert np.array_equal(np.nan_to_num(y[0]), np.nan_to_num(y[-1]))
        assert a[1][2] == 0 and a[1][3] == 0 and a[2][2] == 1
        seen |= set(a[2].tolist())
    gv.close()
    assert {0, 1} <= seen
