"""Incidence, change of basis and the forest, at sizes where the lists and
the scans change shape: one element; fewer elements than a warp; lists longer
than 64 entries; elements of very different size in one bucket; more elements
than a scan tile.

Blocks against the FP64 oracle's interpolated blocks.  Interpolation carries a
value's rounding (32 u max|c| allowed for the sum over a list, u = 2^-53) into
the coefficients by the norms of its three inverses, so the bar is 32 u max|c|
times their product (6e-13, 6e-12 and 1e-10 for degrees 2, 3 and 4).  The number
of incidence entries against a direct test of supports, and two conversions bit
for bit (the lists are filled in no fixed order and sorted).
"""
import math
import time

import numpy as np
import pytest

torch = pytest.importorskip("torch")

from oracle.oracle import Oracle
from paper_1707_01170_gb300 import lrvol as lv
from paper_1707_01170_gb300.synth import volumes as V
from paper_1707_01170_gb300.synth.lrgen import LRVolume, Stream

pytestmark = pytest.mark.gpu

VOLS = {
    "one element": lambda: V.tensor_product((3, 3, 3), (1, 1, 1)),
    "8 elements": lambda: V.tensor_product((1, 2, 3), (2, 2, 2), ncomp=3),
    "degree 4, lists over 128": lambda: V.refined_ball((4, 4, 4), (3, 3, 3), radii=(0.3,), seed=1),
    "mixed sizes": lambda: V.refined_ball((2, 2, 2), (2, 2, 2), centres=((0.2, 0.3, 0.4),), radii=(0.3, 0.2, 0.12),
                                          ncomp=3, seed=2),
    "scan tiles": lambda: V.tensor_product((1, 1, 1), (17, 16, 15)),
    "flat": lambda: V.tensor_product((2, 1, 1), (40, 1, 1)),
}


def _amplification(deg):
    k = 1.0
    for p in (int(d) for d in deg):
        x = (np.arange(p + 1) + 0.5) / (p + 1)
        B = np.stack([math.comb(p, i) * x ** i * (1 - x) ** (p - i) for i in range(p + 1)], 1)
        k *= np.abs(np.linalg.inv(B)).sum(1).max()
    return k


def _incidence(vol):
    n = 0
    s = vol.knot_slices()
    lo = np.stack([vol.knots[:, q][:, 0] for q in s], 1)
    hi = np.stack([vol.knots[:, q][:, -1] for q in s], 1)
    for b in vol.elem_box:
        n += int(np.all((lo <= b[:3]) & (b[3:] <= hi), axis=1).sum())
    return n


def _half_box():
    return LRVolume(deg=np.array([1, 1, 1]), elem_box=np.array([[0.0, 0, 0, 0.5, 0.5, 0.5]]), knots=np.tile([0.0, 0.0, 1.0], (1, 3)),
                    coef=np.ones((1, 1)), weight=np.ones(1), grid=np.array([2, 2, 2]))


@pytest.mark.parametrize("blocks", [(1, 1, 1), (4, 4, 4), (2, 1, 128), (64, 1, 1), (32, 64, 16)])
@pytest.mark.parametrize("split", [lv.SPLIT_BALANCED, lv.SPLIT_MIDPOINT])
def test_forest_shapes(blocks, split):
    """Look-ups are exact for every shape of the forest and both split rules, on a mesh of three element sizes."""
    vol = V.refined_ball((2, 2, 2), (4, 4, 4), centres=((0.3, 0.4, 0.55),), radii=(0.3, 0.15), seed=2)
    X = Stream(3, 3 * 4000 + 8).take(3 * 4000).reshape(-1, 3)
    X[::3] = np.round(X[::3] * 32) / 32
    gv = lv.Volume(vol).build_accel(blocks, split=split)
    got = gv.lookup(torch.from_numpy(X.astype(np.float32)).cuda()).cpu().numpy().astype(np.uint32)
    st = gv.stats()
    gv.close()
    assert np.array_equal(got, Oracle(vol).lookup(X.astype(np.float32)))
    assert (st["depth_max"] == 0) == (st["n_nodes"] == 0)


def test_forest_accepts_and_refuses_as_it_did():
    """A lone element with gaps around it names every block; overlapping elements are refused."""
    gv = lv.Volume(_half_box()).build_accel((4, 4, 4))
    assert (gv.lookup(torch.rand((100, 3), device="cuda")) == 0).all()
    gv.close()
    v = V.tensor_product((1, 1, 1), (2, 2, 2))
    v.elem_box = np.concatenate([v.elem_box, v.elem_box[:1]])
    gv = lv.Volume(v)
    for blocks in ((1, 1, 1), (4, 4, 4)):
        with pytest.raises(lv.LrvolError) as err:
            gv.build_accel(blocks)
        assert err.value.status == lv.ERR_ARG
    gv.close()


def _boxes(lo, hi, n):
    v = _half_box()
    v.elem_box = np.tile(np.array([[*lo, *hi]], dtype=np.float64), (n, 1))
    return v


@pytest.mark.parametrize("name,lo,hi,n", [("cubes", (0, 0, 0), (1, 1, 1), 8000), ("sheets", (0, 0, 0.5), (1, 1, 0.500001), 20000)])
def test_overlapping_boxes_are_refused_at_once(name, lo, hi, n):
    """Boxes that all meet thousands of blocks (in all 2.1e9 and 8.2e7): refused without visiting those."""
    gv = lv.Volume(_boxes(lo, hi, n))
    t = time.perf_counter()
    with pytest.raises(lv.LrvolError) as err:
        gv.build_accel((64, 64, 64))
    assert err.value.status == lv.ERR_ARG and time.perf_counter() - t < 0.1
    gv.close()


def test_small_forests_start_no_threads():
    """Starting the threads of a large mesh takes ten times as long as a small mesh's forest."""
    gv = lv.Volume(V.tensor_product((1, 1, 1), (2, 2, 2)))

    def best(blocks):
        t = []
        for _ in range(30):
            t0 = time.perf_counter()
            gv.build_accel(blocks)
            t.append(time.perf_counter() - t0)
        return min(t)
    one, many = best((1, 1, 1)), best((16, 16, 16))
    gv.close()
    assert many < 4 * one


@pytest.mark.parametrize("name", list(VOLS))
def test_blocks_and_incidence(name):
    vol = VOLS[name]()
    gv = lv.Volume(vol).to_bezier()
    got = gv.get_bezier()
    want = Oracle(vol).bezier_blocks()
    assert got.shape == want.shape
    assert np.abs(got - want).max() <= 32 * 2.0 ** -53 * _amplification(vol.deg) * np.abs(vol.coef).max()
    assert gv.stats()["incidence_entries"] == _incidence(vol)
    again = gv.to_bezier(lv.STORE_F16).get_bezier()
    gv.close()
    assert np.array_equal(got, again)


@pytest.mark.parametrize("n", [1, 32, 33, 128, 129, 8192, 8193, 1 << 17, (1 << 17) + 1, 1 << 20])
def test_incidence_at_the_edges_of_its_routes(n):
    """One trilinear element among n B-splines, of which every third lies over it."""
    knots = np.tile([0.0, 0.0, 1.0], (n, 3))
    knots[np.arange(n) % 3 != 0, 4:6] = 0.25, 0.5      # in y up to 1/2
    knots[np.arange(n) % 3 != 0, 3] = 0.0
    rng = np.random.default_rng(n)
    vol = LRVolume(deg=np.array([1, 1, 1]), elem_box=np.array([[0.0, 0, 0, 1, 1, 1]]), knots=knots, coef=rng.random((n, 1)),
                   weight=np.ones(n), grid=np.array([1, 1, 1]))
    gv = lv.Volume(vol).to_bezier()
    got, entries = gv.get_bezier()[0, 0], gv.stats()["incidence_entries"]
    gv.close()
    want = np.zeros((2, 2, 2))
    want[0, 0, 0] = math.fsum(vol.coef[::3, 0])
    assert entries == (n + 2) // 3
    assert np.abs(got - want).max() <= 2 * n * 2.0 ** -53 * want.max()     # a sum of n / 3 numbers, one after the other


@pytest.mark.parametrize("n", [12285, 12291, 150_000, 300_000])
def test_long_lists_are_sorted(n):
    """96 trilinear elements under n B-splines each third of which lies over all of them: lists of up to 4,095 and
    4,097 entries, sorted by counting and by bits, and of 50,000 and 100,000, in much less than a second."""
    tp = V.tensor_product((1, 1, 1), (4, 4, 6))
    knots = np.tile([-1.0, 0.0, 1.0], (n, 3))
    knots[np.arange(n) % 3 != 0, 3:6] = -3.0, -2.0, -1.0
    rng = np.random.default_rng(n)
    vol = LRVolume(deg=tp.deg, elem_box=tp.elem_box, knots=knots, coef=rng.random((n, 1)), weight=np.ones(n), grid=tp.grid)
    gv = lv.Volume(vol)
    t = time.perf_counter()
    got = gv.to_bezier().get_bezier()
    t = time.perf_counter() - t
    entries = gv.stats()["incidence_entries"]
    gv.close()
    # over [0, 1]^3 every B-spline that counts is (1 - x)(1 - y)(1 - z): a corner's value, added in list order
    lo, hi = tp.elem_box[:, :3], tp.elem_box[:, 3:]
    x = np.stack([1 - lo, 1 - hi], 1)
    corner = np.einsum("ei,ej,ek->ekji", x[:, :, 0], x[:, :, 1], x[:, :, 2])
    want = math.fsum(vol.coef[::3, 0]) * corner[:, None]
    assert entries == 96 * ((n + 2) // 3) and t < 0.5
    assert np.abs(got - want).max() <= 2 * n * 2.0 ** -53 * want.max()
    again = lv.Volume(vol).to_bezier()
    assert np.array_equal(got, again.get_bezier())     # the order of the sums, and so the bits, do not change
    again.close()


@pytest.mark.parametrize("n", [4, 5, 8, 10])
def test_small_routes_refuse_an_element_without_a_spline(n):
    """n^3 elements (every route) of which the last has no B-spline: refused, and again."""
    vol = V.tensor_product((1, 1, 1), (n,) * 3)
    vol.knots[:, :3] = np.minimum(vol.knots[:, :3], 1 - 1 / n)
    gv = lv.Volume(vol)
    for _ in range(2):
        with pytest.raises(lv.LrvolError) as err:
            gv.to_bezier()
        assert err.value.status == lv.ERR_ARG
        with pytest.raises(lv.LrvolError):
            gv.get_bezier()
    gv.close()


def test_small_volumes_convert_without_the_buckets():
    """The buckets' launches and waits double the time of a small volume's conversion (130 against 57 us)."""
    def best(n):
        gv = lv.Volume(V.tensor_product((1, 1, 1), (n,) * 3))
        t = []
        for _ in range(100):
            t0 = time.perf_counter()
            gv.to_bezier()
            t.append(time.perf_counter() - t0)
        gv.close()
        return min(t)
    assert best(2) < 0.7 * best(11)


def test_more_knot_vectors_than_lanes():
    """One trilinear element under 40 B-splines that differ in x, and 3 x 50 on three axes."""
    for nx, ny, nz in ((40, 1, 1), (5, 5, 6), (1, 33, 2)):
        k = [np.stack([-np.arange(1.0, n + 1), np.zeros(n), np.ones(n)], 1) for n in (nx, ny, nz)]
        q = np.stack(np.meshgrid(*[np.arange(n) for n in (nx, ny, nz)], indexing="ij"), -1).reshape(-1, 3)
        knots = np.concatenate([k[a][q[:, a]] for a in range(3)], axis=1)
        rng = np.random.default_rng(nx)
        vol = LRVolume(deg=np.array([1, 1, 1]), elem_box=np.array([[0.0, 0, 0, 1, 1, 1]]), knots=knots,
                       coef=rng.random((len(q), 3)), weight=rng.random(len(q)), grid=np.array([1, 1, 1]))
        gv = lv.Volume(vol).to_bezier()
        got = gv.get_bezier()[0]
        gv.close()
        # over [0, 1] the B-spline on (-k, 0, 1) is 1 - x: coefficients 1, 0
        want = np.zeros((3, 2, 2, 2))
        want[:, 0, 0, 0] = (vol.weight[:, None] * vol.coef).sum(0)
        assert np.abs(got - want).max() <= 8 * len(q) * 2.0 ** -53 * want.max()


def test_element_without_a_spline_is_refused():
    vol = V.tensor_product((2, 2, 2), (3, 3, 3))
    lo = vol.knots[:, 0]
    keep = lo < lo.max()                       # drop the B-splines that reach furthest right ...
    k = vol.knots.copy()
    k[:, :4] = np.minimum(k[:, :4], 2 / 3)     # ... and cut the others' supports before the last elements
    bad = LRVolume(deg=vol.deg, elem_box=vol.elem_box, knots=k[keep], coef=vol.coef[keep], weight=vol.weight[keep],
                   grid=vol.grid)
    gv = lv.Volume(bad)
    with pytest.raises(lv.LrvolError) as err:
        gv.to_bezier()
    assert err.value.status == lv.ERR_ARG
    with pytest.raises(lv.LrvolError):
        gv.get_bezier()
    gv.close()


def test_signed_zeros_and_knots_below_zero():
    """-0 in boxes, knots and coefficients is 0, and knots below 0 lie below it: the same lists and blocks."""
    k = np.array([[-2.0, -1.0, 0.0, 1.0], [-1.0, 0.0, 1.0, 2.0], [0.0, 1.0, 2.0, 3.0]])
    q = np.stack(np.meshgrid(*[np.arange(3)] * 3, indexing="ij"), -1).reshape(-1, 3)
    coef = np.sin(np.arange(27.0))[:, None]
    coef[::4] = 0.0
    vol = LRVolume(deg=np.array([2, 2, 2]), elem_box=np.array([[0.0, 0, 0, 1, 1, 1]]), knots=k[q].reshape(27, 12), coef=coef,
                   weight=np.ones(27), grid=np.array([1, 1, 1]))
    out = []
    for zero in (0.0, -0.0):
        for a in (vol.elem_box, vol.knots, vol.coef):
            a[a == 0] = zero
        gv = lv.Volume(vol).to_bezier()
        f = torch.rand((64, 3), generator=torch.Generator().manual_seed(2)).cuda()
        out.append((gv.stats()["incidence_entries"], gv.get_bezier(), gv.build_accel((1, 1, 1)).eval(f).cpu(),
                    gv.to_bezier(lv.STORE_F16).eval(f).cpu()))
        gv.close()
    assert out[0][0] == out[1][0] == 27 == _incidence(vol)
    assert all(np.array_equal(a, b) for a, b in zip(out[0][1:], out[1][1:]))
