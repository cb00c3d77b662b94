"""The march's first and last samples, and the head table's repeated layer.

alpha_stop <= 0 composites exactly one sample a ray; an opaque transfer
function ends a ray on its first sample; one-sample rays start and end on the
same sample.  Images against the FP64 oracle at RMSE 1e-4 as elsewhere (the
decisions are FP32 on both sides), counts exact.  Look-ups at coordinate 1 and
on block faces are exact for every shape of the table.
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from oracle.oracle import Oracle
from paper_1707_01170_gb300 import lrvol as lv
from paper_1707_01170_gb300.synth import volumes as V
from paper_1707_01170_gb300.synth.lrgen import Stream

pytestmark = pytest.mark.gpu


def _tf(alpha):
    tf = V.seeded_tf(Stream(77), alpha_max=0.05)
    tf.table = tf.table.astype(np.float32).astype(np.float64)
    if alpha is not None:
        tf.table[:, 3] = alpha
    return tf


@pytest.mark.parametrize("mode,h", [("heuristic", 0.0), ("fixed", 1 / 64), ("fixed", 4.0)])
@pytest.mark.parametrize("alpha,alpha_stop", [(None, 0.0), (None, -1.0), (1.0, 0.99), (1.0, 1.0), (0.0, 0.99), (None, 1.0)])
def test_first_and_last_samples(mode, h, alpha, alpha_stop):
    vol = V.refined_ball((2, 2, 2), (3, 3, 3), radii=(0.3,), seed=3)
    cam, tf = V.orbit_camera(Stream(5), 37, 29), _tf(alpha)
    step = V.StepParams(mode=mode, h=h, xi=1 / 64, alpha_stop=alpha_stop)
    ref, ost = Oracle(vol).render(cam, tf, step)
    gv = lv.Volume(vol).build_accel((4, 4, 4)).to_bezier()
    img, st = gv.render(cam, tf, step).cpu().numpy(), gv.stats()
    gv.close()
    assert float(np.sqrt(np.mean((img - ref) ** 2))) <= 1e-4
    assert st["samples"] == ost["samples"] and st["rays_hit"] == ost["rays_hit"]
    if alpha_stop <= 0 or alpha == 1.0 or h == 4.0:
        assert st["samples"] == st["rays_hit"] > 0


@pytest.mark.parametrize("blocks", [(1, 1, 1), (1, 4, 2), (16, 1, 1), (2, 1, 32), (64, 64, 64)])
def test_lookup_at_the_last_layer(blocks):
    vol = V.refined_ball((2, 2, 2), (3, 3, 3), radii=(0.3,), seed=3)     # faces at sixths: not dyadic
    g = np.concatenate([np.arange(0, 65) / 64, np.arange(1, 6) / 6, [1 - 2.0 ** -24, 1 - 2.0 ** -23]])
    X = np.stack(np.meshgrid(g[::9], g, g[::5], indexing="ij"), -1).reshape(-1, 3)
    X = np.concatenate([X, X[:, [1, 0, 2]], X[:, [2, 0, 1]], np.ones((1, 3))]).astype(np.float32)
    gv = lv.Volume(vol).build_accel(blocks)
    got = gv.lookup(torch.from_numpy(X).cuda()).cpu().numpy().astype(np.uint32)
    gv.close()
    assert np.array_equal(got, Oracle(vol).lookup(X))


@pytest.mark.parametrize("storage", [lv.STORE_F32, lv.STORE_F16, lv.STORE_BF16])
@pytest.mark.parametrize("alpha,alpha_stop", [(None, 0.99), (None, 0.0), (1.0, 0.99), (0.0, 0.99)])
@pytest.mark.parametrize("field,degree,blocks,mode", [
    ("scalar", 3, (4, 4, 4), "fixed"), ("scalar", 3, (64, 64, 64), "learned"), ("scalar", 3, (1, 1, 1), "heuristic"),
    ("scalar", 3, (64, 64, 64), "heuristic"), ("magnitude", 2, (4, 4, 4), "learned"), ("magnitude", 2, (64, 64, 64), "heuristic"),
    ("magnitude", 3, (64, 64, 64), "fixed"), ("magnitude", 3, (4, 4, 4), "heuristic"), ("component", 2, (1, 1, 1), "learned"),
    ("component", 3, (4, 4, 4), "heuristic"), ("component", 2, (64, 64, 64), "fixed")])
def test_two_samples_a_pass(field, degree, blocks, mode, alpha, alpha_stop, storage):
    """A frame above 12 CTAs an SM marches one sample a pass, its parts of at most 4 two (Eq. 4 tricubic scalars two
    always; one: fixed speed but for tricubic BF16, and Eq. 4 speed of a small degree-2 volume): the bits and counts
    of the traced kernel, which takes one, and of each other."""
    vol = V.refined_ball((degree,) * 3, (3, 3, 3), radii=(0.3,), seed=3, ncomp=1 if field == "scalar" else 3)
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    tiles = 12 * sms // 33 + 2                       # 33 bands of 8 rows: 12 CTAs an SM and a little more
    rows = 8 * (4 * sms // tiles)
    cam, tf = V.orbit_camera(Stream(5), 16 * tiles - 3, 8 * 33 - 5), _tf(alpha)
    gv = lv.Volume(vol).build_accel(blocks).to_bezier(storage)
    mult = torch.linspace(0.25, 9.0, gv.n_elem, device="cuda") if mode == "learned" else None
    step = V.StepParams(mode=mode, h=1 / 40, xi=1 / 64, alpha_stop=alpha_stop, field=field, mult=mult)
    whole = gv.render(cam, tf, step).clone()
    st = gv.stats()
    parts, sums = torch.full_like(whole, -1.0), np.zeros(3, dtype=np.int64)
    for r0 in range(0, cam.height, rows):
        gv.render(cam, tf, step, out=parts, row_begin=r0, row_end=min(r0 + rows, cam.height))
        sums += [gv.stats()[c] for c in ("samples", "lookups", "rays_hit")]
    pix = torch.stack(torch.meshgrid(torch.arange(cam.width), torch.arange(cam.height), indexing="xy"), -1)
    _, count, rgba = gv.render_trace(cam, tf, step, pix.reshape(-1, 2).int().cuda(), 1)   # one a pass, always
    gv.close()
    assert torch.equal(whole, parts) and sums.tolist() == [st["samples"], st["lookups"], st["rays_hit"]]
    assert torch.equal(rgba.view_as(whole), whole) and int(count.sum()) == st["samples"]
