"""Performance cases: what programs that use this package have it do.

A case is a dict of plain values; `kind` says which call it is:

  frame   one image of a resident volume (fixed, Eq. 4 or learned steps; plain or gradient-shaded; optionally
          trimmed by a boundary mesh that is ray cast for the same camera first)
  serve   a burst of frame requests on the frame server, over two resident volumes
  probe   field values, element ids or gradients at points
  open    a volume made ready: create, forest, change of basis, its blocks read back
  train   one Adam step of the step network
  labels  one training camera: step labels and features
  lines   a rake of streamlines
  tubes   streamline tubes drawn from polylines

The volumes have the meshes of the package's own workloads (config 1: a tricubic ball refinement; config 2: three
nested shells, tricubic; config 3: flow past a box, triquadratic, 3-vector), with coefficients, cameras, transfer
functions, points, meshes and seeds of their own for every seed.  Meshes are built once per process.
"""
import functools
import math

import numpy as np
import torch

from paper_1707_01170_gb300 import learned as LS
from paper_1707_01170_gb300 import lrvol as lv
from paper_1707_01170_gb300.synth import volumes as V
from paper_1707_01170_gb300.synth.lrgen import LRVolume, Refiner, greville

XI = 1 / 256
VECTOR_FIELDS = ("magnitude", "component")


# ---------------------------------------------------------------------------------------------------------------------
# the cases
# ---------------------------------------------------------------------------------------------------------------------

FRAME = {"kind": "frame", "mesh": "shells", "degree": 3, "storage": "f32", "mode": "heuristic", "field": "scalar",
         "projection": "persp", "width": 1920, "height": 1080, "alpha_stop": 0.99, "shaded": False, "triangles": 0}


def listed():
    return [
        # a thumbnail of a small volume at a fixed step, every ray to its end: latency and the number of blocks count
        dict(FRAME, name="frame-256-fixed", mesh="blob", mode="fixed", projection="ortho", width=256, height=256,
             alpha_stop=1.0),
        # the package's benchmark frame: an interactive view of the MR-like volume
        dict(FRAME, name="frame-1080p-eq4"),
        # the same volume at 4K as it is shown in earnest: FP16 blocks, learned steps from features and the network
        dict(FRAME, name="frame-4k-learned", storage="f16", mode="learned", width=3840, height=2160),
        # a lit close-up inside a simulation's geometry (about 2.4M boundary triangles), BF16 blocks
        dict(FRAME, name="frame-720p-lit-trimmed", storage="bf16", width=1280, height=720, shaded=True,
             triangles=2_400_000),
        # flow speed around an obstacle: 3-vector volume larger than L2, FP16 blocks
        dict(FRAME, name="frame-1080p-speed", mesh="flow", degree=2, storage="f16", field="magnitude"),
        # several viewers at once: small and full-HD frames of a scalar and a vector volume in one burst
        {"name": "serve-burst", "kind": "serve", "small": 8, "large": 2, "storage": "f32"},
        # scattered probes of value and gradient (isosurface projection, feature search), an odd number of them
        {"name": "probe-gradient", "kind": "probe", "mesh": "shells", "degree": 3, "storage": "f32", "what": "gradient",
         "order": "scattered", "points": 1_000_003},
        # loading: from the spline's arrays to a volume that can be rendered, and the Bezier blocks for an exporter
        {"name": "open-shells", "kind": "open", "mesh": "shells", "degree": 3, "storage": "f16", "blocks": 64},
        # the training recipe's step: batch 8,192
        {"name": "train-8192", "kind": "train", "batch": 8192},
        # one camera of the training recipe
        {"name": "labels-180p", "kind": "labels", "mesh": "shells", "degree": 3, "width": 320, "height": 180,
         "tau": 4e-4},
        # a rake of the size that the paper traces (88 to 250 seeds)
        {"name": "lines-250", "kind": "lines", "mesh": "flow", "degree": 2, "storage": "f32", "method": "RK4",
         "rule": "heuristic", "seeds": 250},
        # a dense bundle of tubes over a full-HD image
        {"name": "tubes-1080p", "kind": "tubes", "lines": 4096, "samples": 64, "storage": "f32", "width": 1920,
         "height": 1080},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """A case of the listed kinds' ranges: sizes log-uniform and mostly odd, every storage, degree and option."""
    kind = rng.choice(["frame"] * 5 + ["serve", "probe", "probe", "open", "train", "train", "labels", "lines", "tubes"])
    storage = rng.choice(["f32", "f16", "bf16"])
    mesh = rng.choice(["blob", "shells"])
    if kind == "frame":
        vector = rng.random() < 0.35
        mesh = rng.choice(["blob", "flow"]) if vector else mesh
        degree = {"blob": rng.choice([1, 2, 3]), "shells": 3, "flow": 2}[mesh]
        width = _log_int(rng, 96, 2560)
        height = max(64, min(2160, int(width * rng.uniform(0.45, 1.05))))
        return dict(FRAME, mesh=mesh, degree=degree, storage=storage, width=width, height=height,
                    mode=rng.choice(["fixed", "heuristic", "heuristic", "learned"]),
                    field=rng.choice(VECTOR_FIELDS) if vector else "scalar",
                    projection=rng.choice(["persp", "persp", "ortho"]), alpha_stop=rng.choice([0.95, 0.99, 1.0]),
                    shaded=not vector and rng.random() < 0.3,
                    triangles=_log_int(rng, 500, 2_000_000) if rng.random() < 0.25 else 0)
    if kind == "serve":
        return {"kind": kind, "small": rng.randint(1, 16), "large": rng.randint(0, 2), "storage": storage}
    if kind == "probe":
        what = rng.choice(["gradient", "value", "vector"])
        mesh = rng.choice(["blob", "flow"]) if what == "vector" else mesh
        degree = {"blob": rng.choice([1, 2, 3]), "shells": 3, "flow": 2}[mesh]
        return {"kind": kind, "mesh": mesh, "degree": degree, "storage": storage, "what": what,
                "order": rng.choice(["scattered", "grid"]), "points": _log_int(rng, 100, 2_000_000)}
    if kind == "open":
        return {"kind": kind, "mesh": mesh, "degree": rng.choice([1, 2, 3]) if mesh == "blob" else 3,
                "storage": storage, "blocks": rng.choice([16, 32, 64])}
    if kind == "train":
        return {"kind": kind, "batch": _log_int(rng, 64, 16384)}
    if kind == "labels":
        width = _log_int(rng, 64, 320)
        return {"kind": kind, "mesh": mesh, "degree": rng.choice([1, 2, 3]) if mesh == "blob" else 3, "width": width,
                "height": max(36, width * 9 // 16), "tau": rng.choice([4e-4, 8e-4])}
    if kind == "lines":
        mesh = rng.choice(["blob", "flow"])
        return {"kind": kind, "mesh": mesh, "degree": rng.choice([2, 3]) if mesh == "blob" else 2, "storage": storage,
                "method": rng.choice(["RK2", "RK4", "RKF5"]), "rule": "heuristic", "seeds": _log_int(rng, 32, 16384)}
    return {"kind": kind, "lines": _log_int(rng, 40, 4096), "samples": rng.randint(17, 200), "storage": storage,
            "width": _log_int(rng, 256, 1920), "height": _log_int(rng, 200, 1080)}


# ---------------------------------------------------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------------------------------------------------

SHELL_AXES = np.array([[0.41, 0.38, 0.40], [0.32, 0.35, 0.33], [0.26, 0.24, 0.25]])


def _shell_distance(x):
    r = np.stack([np.sqrt(np.sum(((x - 0.5) / a) ** 2, axis=1)) for a in SHELL_AXES], axis=1)
    return (r - 1.0) * SHELL_AXES.mean(axis=1)


@functools.lru_cache(maxsize=None)
def _mesh(name, degree):
    """The refined mesh's arrays and the Greville points of its B-splines."""
    base, levels = {"blob": (8, 2), "shells": (4, 4), "flow": (6, 5)}[name]
    R = Refiner((degree,) * 3, (base,) * 3, levels, 1)
    for level in range(levels):
        box = R.element_boxes()
        c = 0.5 * (box[:, :3] + box[:, 3:])
        if name == "blob":
            near = np.linalg.norm(c - np.array([0.42, 0.55, 0.48]), axis=1) < (0.25, 0.12)[level]
        elif name == "shells":
            near = np.any(np.abs(_shell_distance(c)) < V.CFG2_BANDS[level], axis=1)
        else:
            near = V.box_distance(c) < V.CFG3_DIST[level]
        R.refine(near)
    vol = R.volume(coef=np.zeros((R.n_basis, 1)), name=name)
    return vol, greville(vol)


def _scalar_coef(rng, mesh, g):
    if mesh == "shells":   # three shells of different height and thickness, and a smooth background
        d = _shell_distance(g)
        amp = np.array([0.55, 0.75, 1.0]) * rng.uniform(0.85, 1.0, 3)
        v = np.sum(amp * np.exp(-0.5 * (d / rng.uniform(0.01, 0.02, 3)) ** 2), axis=1)
        for _ in range(8):
            v += 0.015 * np.sin(2 * np.pi * (g @ rng.integers(-3, 4, 3)) + rng.uniform(0, 2 * np.pi))
    else:                  # four Gaussians
        v = np.zeros(len(g))
        for _ in range(4):
            c, s, a = rng.uniform(0.15, 0.85, 3), rng.uniform(0.1, 0.2), rng.uniform(0.5, 1.0)
            v += a * np.exp(-np.sum((g - c) ** 2, axis=1) / (2 * s * s))
    return ((v - v.min()) / (v.max() - v.min()))[:, None]


def _vector_coef(rng, g):
    """Wind along x past the box obstacle (at rest inside it), with four swirls."""
    v = np.tile(np.array([1.0, 0.0, 0.0]), (len(g), 1))
    for _ in range(4):
        c, ax, core = rng.uniform(0.1, 0.9, 3), rng.normal(size=3), rng.uniform(0.04, 0.1)
        ax /= np.linalg.norm(ax)
        r = np.cross(ax, g - c)
        v += rng.uniform(-0.5, 0.5) / core * r * np.exp(-np.sum(r * r, axis=1, keepdims=True) / (2 * core * core))
    s = np.clip(V.box_distance(g) / 0.03, 0.0, 1.0)
    return v * (s * s * (3 - 2 * s))[:, None]


def _spline(mesh, degree, ncomp, seed):
    m, g = _mesh(mesh, degree)
    rng = np.random.default_rng([seed, 1])
    coef = _vector_coef(rng, g) if ncomp == 3 else _scalar_coef(rng, mesh, g)
    return LRVolume(deg=m.deg, elem_box=m.elem_box, knots=m.knots, coef=coef, weight=m.weight, grid=m.grid, name=mesh)


STORAGE = {"f32": lv.STORE_F32, "f16": lv.STORE_F16, "bf16": lv.STORE_BF16}


def _volume(spline, storage, blocks=64):
    return lv.Volume(spline).build_accel((blocks,) * 3).to_bezier(STORAGE[storage])


def _tf(seed, field="scalar"):
    """Eight random control points and three opacity bands, as the package's workloads have them."""
    rng = np.random.default_rng([seed, 2])
    x, ctrl = np.arange(256) / 255.0, rng.uniform(0, 1, (8, 4)) * np.array([1, 1, 1, 0.02])
    ctrl[0, 3] = 0.0
    table = np.stack([np.interp(x, np.linspace(0, 1, 8), ctrl[:, c]) for c in range(4)], axis=1)
    for centre in (0.5, 0.7, 0.95):
        w = np.clip(1.0 - np.abs(x - centre) / 0.04, 0.0, 1.0)[:, None]
        table[:, 3:] = np.maximum(table[:, 3:], rng.uniform(0.05, 0.3) * w)
        table[:, :3] = (1 - w) * table[:, :3] + w * rng.uniform(0, 1, 3)
    lo, hi = {"scalar": (0.0, 1.0), "magnitude": (0.0, 1.5), "component": (-0.5, 1.5)}[field]
    return V.TransferFunction(table=table.astype(np.float32).astype(np.float64), vmin=lo, vmax=hi)


def _camera(seed, width, height, projection="persp"):
    """A view of the whole cube from a random side."""
    rng = np.random.default_rng([seed, 3])
    az, el = rng.uniform(0, 2 * np.pi), rng.uniform(-0.5, 0.5)
    d = np.array([np.cos(el) * np.cos(az), np.cos(el) * np.sin(az), np.sin(el)])
    return V.Camera(projection, int(width), int(height), eye=tuple(0.5 + 1.8 * d), target=(0.5, 0.5, 0.5),
                    up=(0.0, 0.0, 1.0), fovy=math.radians(40.0), extent=1.6)


def _boundary(seed, triangles):
    """A closed mesh of about that many triangles inside the cube."""
    n = max(4, int(math.sqrt(triangles / 4)))
    rng = np.random.default_rng([seed, 4])
    return V.uv_sphere(tuple(0.5 + rng.uniform(-0.05, 0.05, 3)), rng.uniform(0.3, 0.4), n, 2 * n).astype(np.float32)


def _step_model(seed, volume, cam, tf, step):
    """A step network that answers over the range a trained one does: random hidden layers, the output layer scaled to
    log2 multipliers of mean 1.4 and standard deviation 0.8 on the volume's own features."""
    p = LS.init_params(seed)
    model = LS.StepModel(p, LS.TrainConfig(seed=seed))
    f = lv.features(volume, cam, tf, step)
    rows = f[:: max(1, f.shape[0] // 4096)].double()
    y = _network64(model.params.double(), rows)
    model.params[-65:-1] *= float(0.8 / y.std())
    model.params[-1] = 1.4 + model.cfg.margin - float(y.mean() * (0.8 / y.std()))
    model.packed   # packed once, as a program that renders many frames has it
    return model


def _points(seed, n, order):
    gen = torch.Generator(device="cuda").manual_seed(seed)
    if order == "scattered":
        return torch.rand((n, 3), generator=gen, device="cuda")
    # the first n cell centres of a regular grid, x fastest, in a random sub-box (a resampling)
    m = int(math.ceil(n ** (1 / 3)))
    lo = 0.3 * torch.rand(3, generator=gen, device="cuda")
    q = torch.arange(n, device="cuda")
    ijk = torch.stack([q % m, (q // m) % m, q // (m * m)], dim=1)
    return (lo + (ijk + 0.5) * (0.7 / m)).float().contiguous()


def _polylines(seed, lines, samples):
    """Lines as the tracer leaves them: along x with swirls, of different lengths, 32 bytes a sample."""
    rng = np.random.default_rng([seed, 5])
    s = np.arange(samples)[None, :]
    h = rng.uniform(0.002, 0.008, (lines, 1))
    pos = rng.uniform([0.02, 0.05, 0.05], [0.3, 0.95, 0.95], (lines, 3))[:, None, :].repeat(samples, axis=1)
    rad, w, ph = rng.uniform(0.0, 0.03, (lines, 1)), rng.uniform(5, 40, (lines, 1)), rng.uniform(0, 6.28, (lines, 1))
    pos[:, :, 0] += h * s
    pos[:, :, 1] += rad * np.sin(w * h * s + ph)
    pos[:, :, 2] += rad * np.cos(w * h * s + ph)
    out = np.concatenate([np.clip(pos, 0.0, 1.0), (h * s)[:, :, None]], axis=2)
    count = rng.integers(0, samples + 1, lines)
    count[rng.random(lines) < 0.7] = samples
    return torch.from_numpy(out).cuda(), torch.from_numpy(count.astype(np.int32)).cuda()


def _seeds(seed, n):
    rng = np.random.default_rng([seed, 6])
    return torch.from_numpy(rng.uniform([0.02, 0.05, 0.02], [0.10, 0.95, 0.60], (n, 3))).cuda()


LINE_SAMPLES = 1024
LINE_T_END = 1.2


def _rule_step(case):
    return V.StepParams(mode="heuristic", xi=XI, alpha_stop=case.get("alpha_stop", 0.99), field=case.get("field", "scalar"))


def prepare(case, seed):
    kind = case["kind"]
    s = {"case": case}
    if kind == "frame":
        vector = case["field"] in VECTOR_FIELDS
        s["volume"] = _volume(_spline(case["mesh"], case["degree"], 3 if vector else 1, seed), case["storage"])
        s["tf"], s["cam"] = _tf(seed, case["field"]), _camera(seed, case["width"], case["height"], case["projection"])
        s["step"] = V.StepParams(mode=case["mode"], h=XI, xi=XI, alpha_stop=case["alpha_stop"], field=case["field"],
                                 component=0, shading="gradient" if case["shaded"] else "none")
        if case["mode"] == "learned":
            s["rule"] = _rule_step(case)
            s["model"] = _step_model(seed, s["volume"], s["cam"], s["tf"], s["rule"])
        if case["triangles"]:
            s["mesh"] = torch.from_numpy(_boundary(seed, case["triangles"])).cuda()
    elif kind == "serve":
        s["volumes"] = [_volume(_spline("shells", 3, 1, seed), case["storage"]),
                        _volume(_spline("flow", 2, 3, seed), case["storage"])]
        tfs = [_tf(seed), _tf(seed, "magnitude")]
        steps = [V.StepParams(mode="heuristic", xi=XI, alpha_stop=0.99, field=f) for f in ("scalar", "magnitude")]
        sizes = [(1920, 1080)] * case["large"] + [(256, 256)] * case["small"]
        s["requests"] = [(s["volumes"][k % 2], _camera(seed * 1000 + k, *size), tfs[k % 2], steps[k % 2])
                         for k, size in enumerate(sizes)]
        s["server"] = lv.Server(slots=8, arena_bytes=sum(w * h * 16 + 256 for w, h in sizes))
        s["server"].set_priority_pixels(1 << 20)
    elif kind == "probe":
        s["volume"] = _volume(_spline(case["mesh"], case["degree"], 3 if case["what"] == "vector" else 1, seed),
                              case["storage"])
        s["points"] = _points(seed, case["points"], case["order"])
    elif kind == "open":
        s["spline"] = _spline(case["mesh"], case["degree"], 1, seed)
    elif kind == "train":
        # mid-training: random features and targets of the right ranges, moments of earlier steps
        n, gen = case["batch"], torch.Generator(device="cuda").manual_seed(seed)
        s["x"] = 2 * torch.rand((n, 16), generator=gen, device="cuda") - 0.5
        s["target"] = 3 * torch.rand(n, generator=gen, device="cuda")
        s["params"] = torch.from_numpy(LS.init_params(seed)).cuda()
        s["m"] = 1e-2 * torch.randn(lv.MLP_PARAMS, generator=gen, device="cuda")
        s["v"] = 1e-3 * (0.5 + torch.rand(lv.MLP_PARAMS, generator=gen, device="cuda"))
        s["scratch"], s["loss"] = lv.mlp_scratch(n), torch.zeros(1, device="cuda")
    elif kind == "labels":
        s["volume"] = _volume(_spline(case["mesh"], case["degree"], 1, seed), "f32")
        s["tf"], s["cam"], s["step"] = _tf(seed), _camera(seed, case["width"], case["height"]), _rule_step(case)
    elif kind == "lines":
        s["volume"] = _volume(_spline(case["mesh"], case["degree"], 3, seed), case["storage"], 256)
        n = case["seeds"]
        s["seeds"] = _seeds(seed, n)
        # the tracer writes a line's own samples only: a program that reads whole buffers clears them once
        s["out"] = (torch.zeros((n, LINE_SAMPLES, 4), dtype=torch.float64, device="cuda"),
                    torch.zeros(n, dtype=torch.int32, device="cuda"), torch.zeros(n, dtype=torch.int32, device="cuda"))
    elif kind == "tubes":
        s["volume"] = _volume(_spline("flow", 2, 3, seed), case["storage"])
        s["samples"], s["count"] = _polylines(seed, case["lines"], case["samples"])
        s["cam"], s["tf"] = _camera(seed, case["width"], case["height"]), _tf(seed, "magnitude")
    return s


# ---------------------------------------------------------------------------------------------------------------------
# the calls
# ---------------------------------------------------------------------------------------------------------------------

def run(s):
    case = s["case"]
    kind = case["kind"]
    if kind == "frame":
        out, step, cam, tf = {}, s["step"], s["cam"], s["tf"]
        if "model" in s:
            out["mult"] = s["model"].multipliers(s["volume"], cam, tf, s["rule"])
        if "mesh" in s:
            out["trim"] = lv.trim(cam, s["mesh"])
        if out:
            step = V.StepParams(mode=step.mode, h=step.h, xi=step.xi, alpha_stop=step.alpha_stop, field=step.field,
                                component=step.component, shading=step.shading, mult=out.get("mult"),
                                trim=out.get("trim"))
        out["image"] = s["volume"].render(cam, tf, step)
        return out
    if kind == "serve":
        srv = s["server"]
        tickets = [srv.submit(*r) for r in s["requests"]]
        srv.drain()
        images = [srv.image(t) for t in tickets]
        srv.poll()
        for t in tickets:
            srv.release(t)
        return {"images": images}
    if kind == "probe":
        if case["what"] == "gradient":
            return {"gradient": s["volume"].eval_grad(s["points"])}
        return {"element": s["volume"].lookup(s["points"]), "value": s["volume"].eval(s["points"])}
    if kind == "open":
        return {"blocks": _volume(s["spline"], case["storage"], case["blocks"]).get_bezier()}
    if kind == "train":
        lv.mlp_train_step(s["x"], s["target"], s["params"], s["m"], s["v"], 500, 1e-3, s["scratch"], s["loss"])
        return {"params": s["params"], "m": s["m"], "v": s["v"], "loss": s["loss"]}
    if kind == "labels":
        return {"labels": lv.labels(s["volume"], s["cam"], s["tf"], s["step"], 1 / 2048, case["tau"], LS.CAND),
                "features": lv.features(s["volume"], s["cam"], s["tf"], s["step"])}
    if kind == "lines":
        samples, count, status = lv.streamlines(s["volume"], s["seeds"], case["method"], case["rule"], 1.0, LINE_T_END,
                                                max_samples=LINE_SAMPLES, out=s["out"])
        return {"samples": samples, "count": count, "status": status}
    return {"image": lv.tubes(s["volume"], s["cam"], s["samples"], s["count"], 0.002, s["tf"])}


# ---------------------------------------------------------------------------------------------------------------------
# what a pass cannot do without
# ---------------------------------------------------------------------------------------------------------------------

# composited samples a pixel of the whole-cube views above, as measured (Eq. 4 steps at the mesh's largest degree, and
# fixed steps), and Eq. 4 samples a line
SAMPLES_PER_PIXEL = {("blob", "fixed"): 90, ("blob", "heuristic"): 55, ("shells", "fixed"): 88,
                     ("shells", "heuristic"): 140, ("flow", "fixed"): 68, ("flow", "heuristic"): 25}
SAMPLES_PER_LINE = {"flow": 235, "blob": 120}
TRIMMED, LEARNED = 0.2, 0.4   # share of the samples that is left


def _samples(case):
    n = case["width"] * case["height"] * SAMPLES_PER_PIXEL[case["mesh"], "fixed" if case["mode"] == "fixed" else "heuristic"]
    if case["mode"] != "fixed" and case["mesh"] == "blob":
        n /= 2 ** (3 - case["degree"])   # Eq. 4: twice the step for each degree less
    return n * (TRIMMED if case["triangles"] else 1) * (LEARNED if case["mode"] == "learned" else 1)


def _block_bytes(case, ncomp):
    per = 4 if case.get("storage", "f32") == "f32" else 2
    return per * ncomp * (case["degree"] + 1) ** 3 + (0 if per == 4 else 32)


def _sample_flops(degree, ncomp, shaded=False):
    n = degree + 1
    return 49 + 3 * (2 * degree + 1) + ncomp * 2 * (n ** 3 + n ** 2 + n) + (2 * (n ** 3 + 2 * n * n + 3 * n) if shaded else 0)


def work(case):
    kind = case["kind"]
    if kind == "frame":
        elems = _mesh(case["mesh"], case["degree"])[0].n_elem
        ncomp = 3 if case["field"] == "magnitude" else 1
        pixels = case["width"] * case["height"]
        b = elems * (_block_bytes(case, ncomp) + 64) + 16 * pixels + (36 * case["triangles"] + 8 * pixels if case["triangles"] else 0)
        f = _samples(case) * _sample_flops(case["degree"], ncomp, case["shaded"])
        if case["mode"] == "learned":
            f, b = f + elems * 18.6e3, b + elems * 4
        return {"bytes": b, "flops": f}
    if kind == "serve":
        frames = [work(dict(FRAME, storage=case["storage"], width=w, height=h, **which))
                  for k, (w, h) in enumerate([(1920, 1080)] * case["large"] + [(256, 256)] * case["small"])
                  for which in ([{}, {"mesh": "flow", "degree": 2, "field": "magnitude"}][k % 2],)]
        return {key: sum(f[key] for f in frames) for key in ("bytes", "flops")}
    if kind == "probe":
        ncomp = 3 if case["what"] == "vector" else 1
        elems = _mesh(case["mesh"], case["degree"])[0].n_elem
        out = 16 if case["what"] == "gradient" else 4 + 4 * ncomp
        return {"bytes": case["points"] * (12 + out) + min(elems, case["points"]) * (_block_bytes(case, ncomp) + 64),
                "flops": case["points"] * _sample_flops(case["degree"], ncomp, case["what"] == "gradient")}
    if kind == "open":
        m, n = _mesh(case["mesh"], case["degree"])[0], (case["degree"] + 1) ** 3
        pairs = m.n_elem * n   # at least (p+1)^3 B-splines meet an element
        return {"bytes": 8 * (m.knots.size + 2 * m.n_basis + m.elem_box.size) + m.n_elem * (8 * n + _block_bytes(case, 1) + 64),
                "flops": pairs * 4 * n}
    if kind == "train":
        return {"bytes": case["batch"] * 68 + 6 * 4 * lv.MLP_PARAMS, "flops": case["batch"] * 6 * 9280}
    if kind == "labels":
        elems = _mesh(case["mesh"], case["degree"])[0].n_elem
        samples = case["width"] * case["height"] * 8 * SAMPLES_PER_PIXEL[case["mesh"], "heuristic"] * 4
        return {"bytes": elems * (_block_bytes(case, 1) + 64 + 68), "flops": samples * _sample_flops(case["degree"], 1)}
    if kind == "lines":
        steps = case["seeds"] * SAMPLES_PER_LINE[case["mesh"]]
        stages = {"RK2": 2, "RK4": 4, "RKF5": 6}[case["method"]]
        return {"bytes": steps * 32 + case["seeds"] * 32, "flops": steps * stages * (40 + _sample_flops(case["degree"], 3))}
    pixels = case["width"] * case["height"]
    segments = int(0.85 * case["lines"] * case["samples"])
    return {"bytes": segments * 32 + 16 * pixels, "flops": segments * 600 + pixels * 600}


def tolerance(case):
    kind = case["kind"]
    if kind in ("frame", "serve"):
        if case.get("mode") == "learned":
            # the network's operands are BF16: another order of its sums moves some activations by a BF16 step, and
            # with them the lengths of an element's steps
            return {"rel": 1e-2, "max": 0.3}
        # the samples' places are FP32 decisions; what is left is FP32 evaluation, transfer function and compositing
        # (1 - alpha in FP32 before its logarithm: up to 1.2e-5 seen), and the 16-bit blocks' storage (6e-5, 3e-4 seen)
        return {"rel": {"f32": 5e-5, "f16": 2.5e-4, "bf16": 1.3e-3}[case["storage"]], "max": 0.05}
    if kind == "probe":
        return {"rel": {"f32": 3e-6, "f16": 1e-3, "bf16": 8e-3}[case["storage"]], "max": 0.1}
    if kind == "open":
        return {"rel": 2e-13, "max": 1e-10}
    if kind == "train":
        return {"rel": 3e-6, "max": 1e-3}
    if kind == "labels":
        # a label is the outcome of comparisons of FP32 composites
        return {"rel": 2e-5, "max": 0.2, "differ": 5e-3}
    if kind == "lines":
        # a point that falls on the other side of an element's face takes another step from there on
        return {"rel": 1e-4, "max": 0.3, "differ": 5e-3}
    return {"rel": 2e-5, "max": 0.1}   # which segment a pixel shows is an FP32 decision


# ---------------------------------------------------------------------------------------------------------------------
# 64-bit answers in plain torch
#
# Where a sample lies, which element holds it and how far the next one is are FP32 decisions with a stated order of
# operations (include/lrvol.h); they are taken as stated.  Everything computed at the samples is 64-bit.
# ---------------------------------------------------------------------------------------------------------------------

def _fma32(a, b, c):
    return (a.double() * b.double() + c.double()).float()


def _round_up32(x):
    f = x.astype(np.float32)
    return np.where(f.astype(np.float64) < x, np.nextafter(f, np.float32(np.inf)), f)


class _Field64:
    """Bernstein blocks of a spline by interpolation, and element look-up on the finest grid."""

    def __init__(self, spline):
        p = int(spline.deg[0])
        n, self.p, self.ncomp = p + 1, p, spline.coef.shape[1]
        box = torch.from_numpy(spline.elem_box).cuda()
        knots = torch.from_numpy(spline.knots).cuda().reshape(-1, 3, p + 2)
        wc = torch.from_numpy(spline.weight[:, None] * spline.coef).cuda()
        self.lo, self.side = box[:, :3].contiguous(), (box[:, 3:] - box[:, :3]).contiguous()
        nodes = (torch.arange(n, device="cuda", dtype=torch.float64) + 0.5) / n
        vals = torch.zeros((len(box), self.ncomp, n ** 3), dtype=torch.float64, device="cuda")
        lo_s, hi_s = knots[:, :, 0], knots[:, :, -1]
        cell = torch.clamp((0.5 * (box[:, :3] + box[:, 3:]) * 8).long(), 0, 7)
        cell = (cell[:, 2] * 8 + cell[:, 1]) * 8 + cell[:, 0]
        for c in torch.unique(cell).tolist():
            els = torch.nonzero(cell == c)[:, 0]
            blo, bhi = box[els, :3], box[els, 3:]
            near = torch.nonzero(((lo_s < bhi.max(0)[0]) & (hi_s > blo.min(0)[0])).all(1))[:, 0]
            inside = torch.ones((len(els), len(near)), dtype=torch.bool, device="cuda")
            for a in range(3):
                inside &= lo_s[near, a][None] <= blo[:, a][:, None]
                inside &= hi_s[near, a][None] >= bhi[:, a][:, None]
            pairs = torch.nonzero(inside)
            for part in torch.split(pairs, 400_000):
                e, i = els[part[:, 0]], near[part[:, 1]]
                uni = []
                for a in range(3):
                    x = self.lo[e, a][:, None] + self.side[e, a][:, None] * nodes
                    uni.append(self._bspline(knots[i, a], x, p))
                t = torch.einsum("pk,pj,pi->pkji", uni[2], uni[1], uni[0]).reshape(len(part), 1, -1)
                vals.index_add_(0, e, t * wc[i][:, :, None])
        # values at the nodes -> Bernstein coefficients, one axis after the other
        q = np.array([[math.comb(p, i) * ((m + 0.5) / n) ** i * (1 - (m + 0.5) / n) ** (p - i) for i in range(n)] for m in range(n)])
        inv = torch.from_numpy(np.linalg.inv(q)).cuda()
        b = vals.reshape(-1, self.ncomp, n, n, n)
        self.blocks = torch.einsum("zi,yj,xk,ecijk->eczyx", inv, inv, inv, b)
        # element ids on the grid of the finest lines
        G = [int(v) for v in spline.grid]
        ib = np.rint(spline.elem_box * np.array(G * 2)).astype(np.int64)
        ids = np.zeros(G[::-1], dtype=np.int32)
        sizes = ib[:, 3:] - ib[:, :3]
        for size in np.unique(sizes, axis=0):
            sel = np.nonzero((sizes == size).all(1))[0]
            for dz in range(size[2]):
                for dy in range(size[1]):
                    for dx in range(size[0]):
                        ids[ib[sel, 2] + dz, ib[sel, 1] + dy, ib[sel, 0] + dx] = sel
        self.G, self.ids = G, torch.from_numpy(ids).cuda()
        self.faces = [torch.from_numpy(_round_up32(np.arange(1, g) / g)).cuda() for g in G]
        self.ds = torch.from_numpy((2.0 ** -p * (spline.elem_box[:, 3:] - spline.elem_box[:, :3]).min(1)).astype(np.float32)).cuda()
        self.binom = torch.tensor([math.comb(p, i) for i in range(n)], dtype=torch.float64, device="cuda")

    @staticmethod
    def _bspline(k, x, p):
        k = k[:, :, None]
        N = [((k[:, j] <= x) & (x < k[:, j + 1])).double() for j in range(p + 1)]
        for r in range(1, p + 1):
            nxt = []
            for j in range(p + 1 - r):
                d0, d1 = k[:, j + r] - k[:, j], k[:, j + r + 1] - k[:, j + 1]
                a = torch.where(d0 > 0, (x - k[:, j]) / torch.where(d0 > 0, d0, 1.0), 0.0)
                b = torch.where(d1 > 0, (k[:, j + r + 1] - x) / torch.where(d1 > 0, d1, 1.0), 0.0)
                nxt.append(a * N[j] + b * N[j + 1])
            N = nxt
        return N[0]

    def locate(self, p32):
        g = [torch.searchsorted(self.faces[a], p32[:, a].contiguous(), right=True) for a in range(3)]
        return self.ids[g[2], g[1], g[0]].long()

    def _basis(self, u):
        i = torch.arange(self.p + 1, device="cuda", dtype=torch.float64)
        v = 1 - u
        b = self.binom * u[..., None] ** i * v[..., None] ** (self.p - i)
        d1 = torch.cat([torch.zeros_like(u)[..., None], i[1:] * u[..., None] ** (i[1:] - 1) * v[..., None] ** (self.p - i[1:])], -1)
        j = self.p - i[:-1]
        d2 = torch.cat([j * u[..., None] ** i[:-1] * v[..., None] ** (j - 1), torch.zeros_like(u)[..., None]], -1)
        return b, self.binom * (d1 - d2)

    def at(self, e, p32, gradient=False, chunk=1 << 20):
        """Components (n, ncomp), and the gradient of component 0 (n, 3)."""
        vals, grads = [], []
        for q in range(0, len(e), chunk):
            ee = e[q:q + chunk]
            u = (p32[q:q + chunk].double() - self.lo[ee]) / self.side[ee]
            b, d = self._basis(u)
            blk = self.blocks[ee]
            ty = torch.einsum("nczyx,nx->nczy", blk, b[:, 0])
            tz = torch.einsum("nczy,ny->ncz", ty, b[:, 1])
            vals.append(torch.einsum("ncz,nz->nc", tz, b[:, 2]))
            if gradient:
                gx = torch.einsum("nzyx,nx,ny,nz->n", blk[:, 0], d[:, 0], b[:, 1], b[:, 2])
                gy = torch.einsum("nzy,ny,nz->n", ty[:, 0], d[:, 1], b[:, 2])
                gz = torch.einsum("nz,nz->n", tz[:, 0], d[:, 2])
                grads.append(torch.stack([gx, gy, gz], 1) / self.side[ee])
        return torch.cat(vals), torch.cat(grads) if gradient else None


def _rays(cam):
    """FP32 origins and directions of all pixels, row by row, and their interval in the cube."""
    f = np.array(cam.target) - np.array(cam.eye)
    f /= np.sqrt(f @ f)
    r = np.cross(f, cam.up)
    r /= np.sqrt(r @ r)
    u = np.cross(r, f)
    ty = math.tan(0.5 * cam.fovy) if cam.projection == "persp" else 0.5 * cam.extent
    tx = ty * cam.width / cam.height
    one = lambda x: torch.tensor(np.float32(x), device="cuda")  # noqa: E731
    i = torch.arange(cam.width, device="cuda").float().repeat(cam.height) + 0.5
    j = torch.arange(cam.height, device="cuda").float().repeat_interleave(cam.width) + 0.5
    a = _fma32(i, one(2 * tx / cam.width), one(-tx))
    b = _fma32(j, one(-2 * ty / cam.height), one(ty))
    persp = cam.projection == "persp"
    at = [_fma32(a, one(r[c]), _fma32(b, one(u[c]), one(f[c] if persp else cam.eye[c]))) for c in range(3)]
    if persp:
        n = torch.sqrt(_fma32(at[0], at[0], _fma32(at[1], at[1], at[2] * at[2])))
        d = torch.stack([x / n for x in at], 1)
        o = torch.tensor(np.float32(cam.eye), device="cuda").expand_as(d)
    else:
        o = torch.stack(at, 1)
        d = torch.tensor(np.float32(f), device="cuda").expand_as(o)
    inv = 1.0 / d
    ta, tb = (0.0 - o) * inv, (1.0 - o) * inv
    flat = d == 0
    tin = torch.where(flat, 0.0, torch.minimum(ta, tb)).amax(1).clamp_min(0.0)
    tout = torch.where(flat, math.inf, torch.maximum(ta, tb)).amin(1)
    hit = (tin < tout) & ~(flat & ((o < 0) | (o > 1))).any(1)
    return o, d, tin, tout, hit


def _image64(field, cam, tf, step, trim=None):
    o, d, tin, tout, hit = _rays(cam)
    out = torch.zeros((cam.height * cam.width, 4), dtype=torch.float64, device="cuda")
    if trim is not None:
        tr = trim.reshape(-1, 2).float()
        hit &= ~(torch.isinf(tr[:, 0]) & (tr[:, 1] == 0))
        tin = torch.where(~torch.isinf(tr[:, 0]), torch.maximum(tin, tr[:, 0]), tin)
        tout = torch.where(tr[:, 1] != 0, torch.minimum(tout, tr[:, 1]), tout)
        hit &= tin < tout
    table = torch.from_numpy(np.asarray(tf.table, dtype=np.float32).astype(np.float64)).cuda()
    delta = torch.cat([table[1:] - table[:-1], torch.zeros_like(table[:1])])
    px = torch.nonzero(hit)[:, 0]
    o, d, tin, tout = (x[px] for x in (o, d, tin, tout))
    t, C, Tr, k = tin.clone(), torch.zeros((len(px), 3), dtype=torch.float64, device="cuda"), torch.ones(len(px), dtype=torch.float64, device="cuda"), 0
    while len(px):
        p = _fma32(t[:, None], d, o).clamp(0.0, 1.0)
        e = field.locate(p)
        tn = _fma32(torch.tensor(float(k + 1), device="cuda"), torch.tensor(np.float32(step.h), device="cuda"), tin) if step.mode == "fixed" else t + field.ds[e]
        tn = torch.where(tn > t, tn, torch.nextafter(t, torch.full_like(t, math.inf)))
        seg = (torch.minimum(tn, tout) - t).double()
        v, g = field.at(e, p, step.shading == "gradient")
        v = v.square().sum(1).sqrt() if step.field == "magnitude" else v[:, step.component if step.field == "component" else 0]
        x = ((v - tf.vmin) / (tf.vmax - tf.vmin)).clamp(0, 1) * 255
        q = x.floor()
        src = table[q.long()] + (x - q)[:, None] * delta[q.long()]
        T = (1 - src[:, 3]).clamp_min(0) ** (seg / step.xi)
        w = (1 - T) * Tr
        if g is not None:
            light = g.mul(d.double()).sum(1).abs() / g.square().sum(1).sqrt().clamp_min(1e-3 * (tf.vmax - tf.vmin))
            w = w * light.clamp_min(0.4)
        C = C + w[:, None] * src[:, :3]
        Tr = Tr * T
        k += 1
        t = tn
        done = (Tr <= 1 - step.alpha_stop) | ~(t < tout)
        if bool(done.any()):
            out[px[done]] = torch.cat([C[done], 1 - Tr[done, None]], 1)
            keep = ~done
            px, o, d, tin, tout, t, C, Tr = (x[keep] for x in (px, o, d, tin, tout, t, C, Tr))
    return out.reshape(cam.height, cam.width, 4)


def _pairs(i0, i1, j0, j1, width):
    """(primitive, pixel) for every pixel of each primitive's box, in parts."""
    w = (i1 - i0 + 1).clamp_min(0)
    n = w * (j1 - j0 + 1).clamp_min(0)
    first = 0
    ends = torch.cumsum(n, 0)
    while first < len(n):
        base = int(ends[first - 1]) if first else 0
        last = max(first + 1, int(torch.searchsorted(ends, base + 4_000_000, right=True)))
        k = torch.repeat_interleave(torch.arange(first, last, device="cuda"), n[first:last])
        q = torch.arange(len(k), device="cuda") - (ends[k] - n[k] - base)
        yield k, (j0[k] + q // w[k]) * width + i0[k] + q % w[k]
        first = last


def _pixel_boxes(cam, lo, hi):
    """Pixel boxes, a pixel wide of the exact ones, of boxes in front of the eye (corners lo, hi)."""
    f = np.array(cam.target) - np.array(cam.eye)
    f /= np.sqrt(f @ f)
    r = np.cross(f, cam.up)
    r /= np.sqrt(r @ r)
    u = np.cross(r, f)
    persp = cam.projection == "persp"
    ty = math.tan(0.5 * cam.fovy) if persp else 0.5 * cam.extent
    tx = ty * cam.width / cam.height
    frame = torch.from_numpy(np.stack([r, u, f], 1)).cuda()
    eye = torch.tensor(cam.eye, dtype=torch.float64, device="cuda")
    xs, ys = [], []
    for c in range(8):
        q = torch.stack([(hi if c >> a & 1 else lo)[:, a] for a in range(3)], 1) - eye
        z = q @ frame
        s = z[:, 2] if persp else 1.0
        xs.append((z[:, 0] / s + tx) * cam.width / (2 * tx) - 0.5)
        ys.append((ty - z[:, 1] / s) * cam.height / (2 * ty) - 0.5)
    xs, ys = torch.stack(xs), torch.stack(ys)
    clip = lambda v, m: v.clamp(-2, m + 1).long()  # noqa: E731
    return (clip(xs.amin(0).floor() - 1, cam.width).clamp_min(0), clip(xs.amax(0).ceil() + 1, cam.width).clamp_max(cam.width - 1),
            clip(ys.amin(0).floor() - 1, cam.height).clamp_min(0), clip(ys.amax(0).ceil() + 1, cam.height).clamp_max(cam.height - 1))


def _trim64(cam, tris):
    o, d, _, _, _ = _rays(cam)
    v = torch.from_numpy(tris).cuda().double().reshape(-1, 3, 3)
    near = torch.full((len(o),), math.inf, dtype=torch.float64, device="cuda")
    far = torch.zeros(len(o), dtype=torch.float64, device="cuda")
    for k, px in _pairs(*_pixel_boxes(cam, v.amin(1), v.amax(1)), cam.width):
        oo, dd = o[px].double(), d[px].double()
        a, b, c = (v[k, m] - oo for m in range(3))
        U, W_, Q = (torch.cross(x, y, dim=1).mul(dd).sum(1) for x, y in ((c, b), (a, c), (b, a)))
        det = U + W_ + Q
        t = (U[:, None] * a + W_[:, None] * b + Q[:, None] * c).mul(dd).sum(1) / det
        ok = (((U >= 0) & (W_ >= 0) & (Q >= 0)) | ((U <= 0) & (W_ <= 0) & (Q <= 0))) & (det != 0) & (t > 0)
        front = torch.cross(b - a, c - a, dim=1).mul(dd).sum(1) < 0
        near.scatter_reduce_(0, px[ok & front], t[ok & front], "amin")
        far.scatter_reduce_(0, px[ok & ~front], t[ok & ~front], "amax")
    return torch.stack([near, far], 1).reshape(cam.height, cam.width, 2)


def _tubes64(field, cam, samples, count, radius, tf):
    o, d, _, _, _ = _rays(cam)
    n, m = samples.shape[:2]
    line = torch.arange(n, device="cuda").repeat_interleave(m - 1)
    k = torch.arange(m - 1, device="cuda").repeat(n)
    ok = k < count.long()[line] - 1
    line, k = line[ok], k[ok]
    a, b = samples[line, k, :3].float(), samples[line, k + 1, :3].float()
    best = torch.full((len(o),), math.inf, device="cuda")
    radius = torch.tensor(np.float32(radius), device="cuda")

    def dot(x, y):
        return (x[:, 0] * y[:, 0] + x[:, 1] * y[:, 1]) + x[:, 2] * y[:, 2]

    def hits(s, px):   # in FP32, every operation rounded
        dd, ba, oa, ob = d[px], b[s] - a[s], o[px] - a[s], o[px] - b[s]
        baba, bard, baoa, rdoa = dot(ba, ba), dot(ba, dd), dot(ba, oa), dot(dd, oa)
        A = baba - bard * bard
        B = baba * rdoa - baoa * bard
        H = B * B - A * ((baba * dot(oa, oa) - baoa * baoa) - radius * radius * baba)
        tb = (-B - H.clamp_min(0).sqrt()) / A
        y = baoa + tb * bard
        body = (A > 0) & (H >= 0) & (y > 0) & (y < baba)
        t = torch.where(body & (tb > 0), tb, math.inf)
        for x in (oa, ob):
            p = dot(dd, x)
            h = p * p - (dot(x, x) - radius * radius)
            tc = -p - h.clamp_min(0).sqrt()
            t = torch.where(~body & (h > 0) & (tc > 0), torch.minimum(t, tc), t)
        return t

    boxes = _pixel_boxes(cam, (torch.minimum(a, b) - radius).double(), (torch.maximum(a, b) + radius).double())
    for s, px in _pairs(*boxes, cam.width):
        best.scatter_reduce_(0, px, hits(s, px), "amin")
    seg = torch.full((len(o),), len(a), dtype=torch.int64, device="cuda")
    for s, px in _pairs(*boxes, cam.width):
        t = hits(s, px)
        won = torch.isfinite(t) & (t == best[px])
        seg.scatter_reduce_(0, px[won], s[won], "amin")
    out = torch.zeros((len(o), 4), dtype=torch.float64, device="cuda")
    px = torch.nonzero(torch.isfinite(best))[:, 0]
    s = seg[px]
    p = o[px].double() + best[px, None].double() * d[px].double()
    ba, q = (b[s] - a[s]).double(), a[s].double()
    h = ((p - q).mul(ba).sum(1) / ba.square().sum(1).clamp_min(1e-300)).clamp(0, 1)
    q = q + h[:, None] * ba
    q32 = q.float()
    v, _ = field.at(field.locate(q32), q32)
    x = ((v.square().sum(1).sqrt() - tf.vmin) / (tf.vmax - tf.vmin)).clamp(0, 1) * 255
    i = x.floor().clamp_max(254)
    table = torch.from_numpy(np.asarray(tf.table, dtype=np.float32).astype(np.float64)).cuda()
    rgb = table[i.long(), :3] + (x - i)[:, None] * (table[i.long() + 1, :3] - table[i.long(), :3])
    nrm = p - q
    light = (nrm.mul(d[px].double()).sum(1).abs() / nrm.square().sum(1).sqrt()).clamp_min(0.4)
    out[px] = torch.cat([light[:, None] * rgb, torch.ones_like(light)[:, None]], 1)
    return out.reshape(cam.height, cam.width, 4)


def _features64(field, spline, cam, tf):
    w, ctr = field.side, field.lo + 0.5 * field.side
    blk = field.blocks.reshape(len(w), field.ncomp, -1)
    x = [(v.reshape(-1) - tf.vmin) / (tf.vmax - tf.vmin) for v in (blk.amin(2), blk.amax(2))]
    table = np.asarray(tf.table, dtype=np.float32).astype(np.float64)
    i0 = (255 * x[0].clamp(0, 1)).floor().long().cpu().numpy()
    i1 = np.minimum(255, (255 * x[1].clamp(0, 1)).ceil().long().cpu().numpy())
    stat = np.zeros((256, 256, 4))   # max alpha, mean alpha, slope, colour range over entries i .. j
    for i in range(256):
        a, c = table[i:, 3], table[i:, :3]
        stat[i, i:, 0] = np.maximum.accumulate(a)
        stat[i, i:, 1] = np.cumsum(a) / np.arange(1, len(a) + 1)
        stat[i, i:, 2] = 255 * np.maximum.accumulate(np.concatenate([[0.0], np.abs(np.diff(a))]))
        stat[i, i:, 3] = (np.maximum.accumulate(c, 0) - np.minimum.accumulate(c, 0)).max(1)
    st = torch.from_numpy(stat[i0, i1]).cuda()
    direction = ctr - torch.tensor(cam.eye, dtype=torch.float64, device="cuda")
    direction = direction / direction.square().sum(1, keepdim=True).sqrt()
    ds, dx = field.ds.double(), x[1] - x[0]
    return torch.cat([(64 * w).log2(), torch.stack([x[0], x[1], dx], 1), st, direction, (2048 * ds).log2()[:, None],
                      ((direction.abs() * w).sum(1) / (8 * ds))[:, None], (1 + 255 * dx).log2()[:, None]], 1)


def _network64(p, x):
    """y of the 16-64-64-64-1 network for parameters in the library's order."""
    h, at = x, 0
    for n_in in (16, 64, 64):
        w, b = p[at:at + n_in * 64].reshape(n_in, 64), p[at + n_in * 64:at + n_in * 64 + 64]
        h, at = torch.relu(h @ w + b), at + n_in * 64 + 64
    return h @ p[at:at + 64] + p[at + 64]


def _lines64(field, seeds, method):
    a, b = {"RK2": ([[], [0.5]], [0, 1]), "RK4": ([[], [0.5], [0, 0.5], [0, 0, 1]], [1 / 6, 1 / 3, 1 / 3, 1 / 6]),
            "RKF5": ([[], [1 / 4], [3 / 32, 9 / 32], [1932 / 2197, -7200 / 2197, 7296 / 2197],
                      [439 / 216, -8, 3680 / 513, -845 / 4104], [-8 / 27, 2, -3544 / 2565, 1859 / 4104, -11 / 40]],
                     [16 / 135, 0, 6656 / 12825, 28561 / 56430, -9 / 50, 2 / 55])}[method]
    n = len(seeds)
    out = torch.zeros((n, LINE_SAMPLES, 4), dtype=torch.float64, device="cuda")
    count, status = torch.ones(n, dtype=torch.int32, device="cuda"), torch.full((n,), 2, dtype=torch.int32, device="cuda")
    out[:, 0, :3] = seeds
    live, x, t = torch.arange(n, device="cuda"), seeds.clone(), torch.zeros(n, dtype=torch.float64, device="cuda")
    for k in range(1, LINE_SAMPLES):
        h = torch.minimum(field.ds[field.locate(x.float())].double(), LINE_T_END - t)
        inside, ks = torch.ones(len(x), dtype=torch.bool, device="cuda"), []
        for row in a:
            y = x + h[:, None] * sum((c * q for c, q in zip(row, ks)), torch.zeros_like(x))
            y = y.float()
            inside &= ((y >= 0) & (y <= 1)).all(1)
            ks.append(field.at(field.locate(y.clamp(0, 1)), y.clamp(0, 1))[0])
        x = x + h[:, None] * sum(c * q for c, q in zip(b, ks))
        inside &= ((x.float() >= 0) & (x.float() <= 1)).all(1)
        status[live[~inside]] = 1
        t = t + h
        live, x, t = live[inside], x[inside], t[inside]
        out[live, k, :3], out[live, k, 3] = x, t
        count[live] = k + 1
        ended = t >= LINE_T_END
        status[live[ended]] = 0
        live, x, t = live[~ended], x[~ended], t[~ended]
        if not len(live):
            break
    return {"samples": out, "count": count, "status": status}


def exact(case, seed):
    kind = case["kind"]
    if kind == "train":
        s = prepare(case, seed)
        p = s["params"].double().requires_grad_(True)
        loss = 0.5 * (_network64(p, s["x"].double()) - s["target"].double()).square().mean()
        g, = torch.autograd.grad(loss, p)
        m, v = 0.9 * s["m"].double() + 0.1 * g, 0.999 * s["v"].double() + 0.001 * g * g
        p = p.detach() - 1e-3 * (m / (1 - 0.9 ** 500)) / ((v / (1 - 0.999 ** 500)).sqrt() + 1e-8)
        return {"params": p, "m": m, "v": v, "loss": loss.detach().reshape(1)}
    if kind == "open":
        return {"blocks": _Field64(_spline(case["mesh"], case["degree"], 1, seed)).blocks.cpu().numpy()}
    if kind == "serve":
        fields = [_Field64(_spline("shells", 3, 1, seed)), _Field64(_spline("flow", 2, 3, seed))]
        images = []
        for k, size in enumerate([(1920, 1080)] * case["large"] + [(256, 256)] * case["small"]):
            field = ("scalar", "magnitude")[k % 2]
            step = V.StepParams(mode="heuristic", xi=XI, alpha_stop=0.99, field=field)
            images.append(None if size[0] > 256 else _image64(fields[k % 2], _camera(seed * 1000 + k, *size), _tf(seed, field), step))
        return {"images": images} if case["small"] else None
    if kind == "tubes":
        samples, count = _polylines(seed, case["lines"], case["samples"])
        return {"image": _tubes64(_Field64(_spline("flow", 2, 3, seed)), _camera(seed, case["width"], case["height"]),
                                  samples, count, 0.002, _tf(seed, "magnitude"))}
    vector = kind == "lines" or case.get("what") == "vector" or case.get("field") in VECTOR_FIELDS
    spline = _spline(case["mesh"], case["degree"], 3 if vector else 1, seed)
    field = _Field64(spline)
    if kind == "lines":
        return _lines64(field, _seeds(seed, case["seeds"]), case["method"])
    if kind == "probe":
        pts = _points(seed, case["points"], case["order"])
        e = field.locate(pts)
        v, g = field.at(e, pts, case["what"] == "gradient")
        return {"gradient": torch.cat([v, g], 1)} if g is not None else {"element": e.int(), "value": v}
    if kind == "labels":   # the labels are whole values
        return {"labels": None, "features": _features64(field, spline, _camera(seed, case["width"], case["height"]), _tf(seed))}
    out, cam, tf = {}, _camera(seed, case["width"], case["height"], case["projection"]), _tf(seed, case["field"])
    if case["mode"] == "learned":
        if vector:
            return None
        # the image follows the multipliers that the BF16 network gives, so it has no value of its own
        s = prepare(case, seed)
        y = _network64(s["model"].params.double(), _features64(field, spline, cam, tf)) - s["model"].cfg.margin
        return {"mult": 2.0 ** y.clamp(0.0, 3.0), "image": None}
    if case["triangles"]:
        out["trim"] = _trim64(cam, _boundary(seed, case["triangles"]))
    step = V.StepParams(mode=case["mode"], h=XI, xi=XI, alpha_stop=case["alpha_stop"], field=case["field"],
                        component=0, shading="gradient" if case["shaded"] else "none")
    # a larger image takes too long
    out["image"] = _image64(field, cam, tf, step, out.get("trim")) if case["width"] * case["height"] <= 3_000_000 else None
    return out
