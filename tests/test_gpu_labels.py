"""The label kernel where its loops change shape: one candidate, sixteen, more
candidate samples than lanes; visits of fewer and of many more than 32 fine
samples; images that are not a multiple of a CTA's 2x2 rays; every degree.

A label is the outcome of comparisons err <= tau, FP32 here and FP64 in the
oracle, whose composites differ by about 1e-3 of tau: labels lie between the
oracle's at tau (1 -+ 0.02), and 98 % of them (all of fewer than 50) are equal.
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from oracle.oracle import Oracle
from paper_1707_01170_gb300 import lrvol as lv
from paper_1707_01170_gb300.synth import volumes as V
from paper_1707_01170_gb300.synth.lrgen import Stream

pytestmark = pytest.mark.gpu

CANDS = {"one": (1.0,), "two": (1.0, 8.0), "sixteen": tuple(0.25 * k for k in range(1, 17)), "short": (0.02, 0.05, 1.0)}


@pytest.mark.parametrize("cand", sorted(CANDS))
@pytest.mark.parametrize("deg,h_fine", [(1, 1 / 64), (2, 1 / 512), (3, 1 / 2048)])
def test_labels(deg, h_fine, cand):
    vol = V.refined_ball((deg,) * 3, (3, 3, 3), centres=((0.45, 0.5, 0.55),), radii=(0.35,), seed=9)
    orc = Oracle(vol)
    tf = V.seeded_tf(Stream(31), alpha_max=0.05)
    tf.table = tf.table.astype(np.float32).astype(np.float64)
    cam, tau = V.orbit_camera(Stream(32 + deg), 5, 3), 4e-4
    step = V.StepParams(mode="heuristic", xi=1 / 256, alpha_stop=0.97)
    gv = lv.Volume(vol).build_accel((4, 4, 4)).to_bezier()
    got = lv.labels(gv, cam, tf, step, h_fine, tau, CANDS[cand]).cpu().numpy()
    gv.close()
    want, low, high = (orc.labels(cam, tf, step, h_fine, t, CANDS[cand]) for t in (tau, 0.98 * tau, 1.02 * tau))
    seen = want < len(CANDS[cand])
    assert seen.sum() > 10 and np.array_equal(seen, got < len(CANDS[cand]))
    assert np.all((low <= got) & (got <= high))
    assert (got != want).sum() <= 0.02 * seen.sum()
