"""Performance cases: the calls a user of this framework makes, over the sizes
its workloads cover.

A case is one pass of a render job through the public entry points (`Scene`,
`Cache`, `Cache.render_iteration`, `Cache.update_counts`, `Cache.get_state`):

* kind "iteration" -- one render of a running job on a capturable stream, as
  the loop of a training or rendering program calls it: the next iteration
  index, statistics collected, image statistics updated.  The cache holds what
  such a job has learned: in MARS mode the pixel estimate, per-cell count factors
  and guide distributions.  Those are seeded fields under which the path trees
  have the shape of the workload's own, not learned ones: learned factors
  depend on the order of floating-point atomics in their last bits, which flips
  a stochastic rounding somewhere in millions of vertices, so no two runs would
  have the same inputs.
* kind "train" -- one warm-up training iteration of the bidirectional
  application with its count update, octree refinement and a checkpoint of the
  learned state (counts do not feed back into a warm-up render, so the
  repeated pass is reproducible).
* kind "first_image" -- what a request of the serving stream pays before its
  second iteration: scene (hierarchy build), cache and the first warm-up render
  into a host image, then the release of both.

The outputs are float32 images, counters (whole numbers) and the statistics;
a rendered sample passes through discrete decisions (stochastic rounding,
visibility, the bin a uniform picks), so a 64-bit evaluation of the same
formulas follows other paths: `exact` has no value for a render.
"""
from __future__ import annotations

import math

import numpy as np
import torch

import mars_workloads as W
import paper_2410_20429_gb300 as M
from mars_workloads.scenes import GUIDE_BINS

BSDF, NEE, GUIDED, LIGHT = W.TECH_BSDF, W.TECH_NEE, W.TECH_GUIDED, W.TECH_LIGHT

# What the workloads' learned count factors look like: per technique slot the
# median count at a camera ray's first vertex, the standard deviation of its
# logarithm over the cells and the share of cells whose factor is zero, chosen
# so that the depth waves hold as many rays as in the workload's MARS
# iterations; and the rays a pixel's path tree holds (camera ray and every
# drawn sample).
FIELDS = {
    "box": (((1.7, 0.5, 0.0), (1.2, 0.6, 0.2), (0.0, 0.0, 1.0)), 7.0),
    "room": (((1.5, 0.6, 0.06), (1.6, 0.8, 0.3), (0.9, 0.8, 0.2)), 17.0),
    "heightfield": (((1.7, 0.8, 0.1), (0.4, 1.0, 0.6), (1.4, 0.8, 0.2)), 9.0),
    "large": (((2.6, 0.7, 0.1), (5.0, 0.8, 0.1), (0.0, 0.0, 1.0)), 11.0),
    "bdpt_heightfield": (((3.8, 0.8, 0.06), (0.4, 1.0, 0.6), (0.25, 0.8, 0.2)), 12.0),
    "bdpt_large": (((2.4, 0.7, 0.1), (4.0, 0.8, 0.1), (0.1, 0.8, 0.5)), 10.0),
}
ESTIMATE = 0.1      # median of the pixel estimates
N_ESTIMATE = 4096   # renders the estimate stands for: the timed ones hardly move it
# node visits and primitive tests of a ray in such a scene (a binary hierarchy
# over one primitive per leaf), for the operations a pass cannot do without
VISITS = {"box": (5, 1.2), "room": (15, 2), "heightfield": (24, 3), "large": (25, 3), "bdpt_heightfield": (24, 3),
          "bdpt_large": (25, 3)}


def listed():
    return [
        # the Cornell-like box at its own size: the smallest job, where a render is a chain of tiny launches
        _it("box_64", "box", 64, 64, D=5, grid=8, tech=BSDF | NEE),
        # an iteration of a served request: small image, many spheres, the server's multiplicity cap
        _it("served_room_128", "room", 128, 128, D=10, grid=15, tech=BSDF | NEE | GUIDED, prims=459, mult=16.0),
        # a request's odd-sized preview by fixed-count MIS, unaware weights, float32 statistics, a dense room
        _it("room_odd_fixed", "room", 317, 203, D=7, grid=19, tech=BSDF | NEE | GUIDED, prims=1500, mode="fixed",
            aware=False, fp32=True),
        # the headline workload's warm-up (one continuation per vertex) ...
        _it("room_512_warmup", "room", 512, 512, D=10, grid=32, tech=BSDF | NEE | GUIDED, prims=64, mode="warmup"),
        # ... and its MARS iterations, with the launch shape autotuned once per job, as the README's loop does
        _it("room_512_mars", "room", 512, 512, D=10, grid=32, tech=BSDF | NEE | GUIDED, prims=64, tune=True),
        # 131k triangles, one hidden emitter, unidirectional with guiding
        _it("heightfield_1024", "heightfield", 1024, 1024, D=10, grid=32, tech=BSDF | NEE | GUIDED, prims=256),
        # 524k triangles and 4096 spheres, unidirectional
        _it("large_2048", "large", 2048, 2048, D=12, grid=32, tech=BSDF | NEE, prims=512),
        # the bidirectional application's two workloads: octree cache, brightest-pixel rejection, combination
        _it("bdpt_heightfield_1024", "bdpt_heightfield", 1024, 1024, D=10, grid=32, tech=BSDF | NEE | LIGHT, prims=256,
            octree=65536),
        _it("bdpt_large_2048", "bdpt_large", 2048, 2048, D=12, grid=32, tech=BSDF | NEE | LIGHT, prims=512, octree=65536),
        # a training iteration with its update and a checkpoint
        {"name": "train_bdpt_checkpoint", "kind": "train", "scene": "bdpt_heightfield", "width": 200, "height": 150,
         "D": 8, "grid": 8, "tech": BSDF | NEE | LIGHT, "prims": 64, "octree": 4096},
        # a served request from its description to its first image
        {"name": "request_first_image", "kind": "first_image", "scene": "room", "width": 256, "height": 256, "D": 10,
         "grid": 24, "tech": BSDF | NEE | GUIDED, "prims": 700, "bvh": 0},
    ]


def _it(name, scene, w, h, *, D, grid, tech, prims=0, mode="mars", aware=True, fp32=False, mult=0.0,
        octree=0, tune=False):
    return {"name": name, "kind": "iteration", "scene": scene, "width": w, "height": h, "D": D, "grid": grid,
            "tech": tech, "prims": prims, "mode": mode, "aware": aware, "fp32": fp32, "mult": mult,
            "octree": octree, "tune": tune}


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """One more case of the listed ranges: any workload at any of its sizes."""
    family = rng.choice(["box", "room", "room", "served", "heightfield", "large", "bdpt_heightfield", "bdpt_large",
                         "train", "first_image"])
    mode = rng.choice(["mars", "mars", "warmup", "fixed"])
    aware = rng.random() < 0.75
    if family == "box":
        c = _it("", "box", _log(rng, 24, 400), _log(rng, 24, 400), D=rng.randint(2, 6), grid=rng.randint(4, 16),
                tech=BSDF | NEE, mode=mode, aware=aware)
    elif family in ("room", "served"):
        served = family == "served"
        hi = 512 if served else 1100
        c = _it("", "room", _log(rng, 48, hi), _log(rng, 48, hi), D=10 if served else rng.randint(3, 10),
                grid=rng.randint(8, 32), tech=rng.choice([BSDF | NEE | GUIDED, BSDF | NEE | GUIDED, BSDF | NEE]),
                prims=_log(rng, 16, 4096), mode="mars" if served else mode, aware=aware or served,
                fp32=not served and rng.random() < 0.2, mult=16.0 if served else 0.0)
    elif family == "heightfield":
        c = _it("", "heightfield", _log(rng, 128, 1024), _log(rng, 128, 1024), D=rng.randint(4, 10),
                grid=rng.randint(12, 32), tech=BSDF | NEE | GUIDED, prims=_log(rng, 40, 256), mode=mode, aware=aware)
    elif family == "large":
        c = _it("", "large", _log(rng, 256, 2000), _log(rng, 256, 2000), D=rng.randint(4, 12),
                grid=rng.randint(16, 32), tech=BSDF | NEE, prims=_log(rng, 128, 512), mode=mode, aware=aware)
    elif family in ("bdpt_heightfield", "bdpt_large"):
        hi = 1024 if family == "bdpt_heightfield" else 2000
        c = _it("", family, _log(rng, 128, hi), _log(rng, 128, hi), D=rng.randint(4, 10 if hi == 1024 else 12),
                grid=rng.choice([16, 32]), tech=BSDF | NEE | LIGHT, prims=_log(rng, 48, 256 if hi == 1024 else 512),
                mode=mode, aware=aware, octree=rng.choice([0, 65536]))
    elif family == "train":
        c = {"kind": "train", "scene": "bdpt_heightfield", "width": _log(rng, 48, 400), "height": _log(rng, 48, 400),
             "D": rng.randint(4, 10), "grid": 8, "tech": rng.choice([BSDF | NEE | LIGHT, BSDF | NEE]),
             "prims": _log(rng, 16, 128), "octree": 4096}
    else:
        res = rng.choice([64, 128, 256, 512])
        c = {"kind": "first_image", "scene": "room", "width": res, "height": res - rng.randint(0, 9), "D": 10,
             "grid": rng.randint(8, 32), "tech": BSDF | NEE | GUIDED, "prims": _log(rng, 16, 4096),
             "bvh": rng.choice([0, 0, 1])}
    c.pop("name", None)
    return c


def _scene(case, seed):
    kind, w, h, n = case["scene"], case["width"], case["height"], case["prims"]
    if kind == "box":
        return W.box_scene(w, h)
    if kind == "room":
        return W.guided_room_scene(seed % 1000003, w, h, n_spheres=n)
    if kind in ("large", "bdpt_large"):
        return W.heightfield_scene(seed % 1000003, n, w, h, n_spheres=8 * n, n_lights=8, ggx_fraction=1.0)
    return W.heightfield_scene(seed % 1000003, n, w, h, n_spheres=max(8, 200 * n // 256))


def _counts(scene, n_cells, seed):
    """Seeded count factors (q_rr, q_s, valid) of the shape FIELDS gives."""
    g = torch.Generator(device="cuda").manual_seed(seed & 0x7FFFFFFF)

    def rand(*shape):
        return torch.rand(*shape, generator=g, device="cuda")

    q_rr = torch.zeros(n_cells, 3, 3, device="cuda")
    for t, (beta, sd, zero) in enumerate(FIELDS[scene][0]):
        mu = math.log(max(beta, 1e-6) * ESTIMATE)
        z = torch.randn(n_cells, 1, generator=g, device="cuda").clamp_(-2.5, 2.5)
        ch = 0.15 * torch.randn(n_cells, 3, generator=g, device="cuda").clamp_(-2.5, 2.5)
        q_rr[:, t] = torch.exp(mu + sd * z + ch) * (rand(n_cells, 1) >= zero)
    q_s = q_rr * (0.75 + 0.24 * rand(n_cells, 3, 1))
    valid = rand(n_cells, 3) < 0.97
    return q_rr.cpu().numpy(), q_s.cpu().numpy(), valid.to(torch.uint8).cpu().numpy()


def _estimate(w, h, seed):
    """A seeded smooth positive image: the pixel estimate of a long-running job."""
    g = torch.Generator(device="cuda").manual_seed((seed + 2) & 0x7FFFFFFF)
    z = sum(a * torch.nn.functional.interpolate(torch.randn(1, 3, n, n, generator=g, device="cuda").clamp_(-2, 2),
                                                size=(h, w), mode="bilinear")
            for a, n in ((0.3, 4), (0.2, 16)))
    z = z + 0.3 * torch.nn.functional.interpolate(torch.randn(1, 1, 8, 8, generator=g, device="cuda").clamp_(-2, 2),
                                                  size=(h, w), mode="bilinear")
    return (ESTIMATE * torch.exp(z))[0].permute(1, 2, 0).reshape(-1, 3).cpu().numpy()


def _guide(n_cells, seed):
    """Seeded guide CDFs: 90 % a sparse histogram with one lobe, 10 % uniform."""
    g = torch.Generator(device="cuda").manual_seed((seed + 1) & 0x7FFFFFFF)
    h = torch.rand(n_cells, GUIDE_BINS, generator=g, device="cuda")
    h = torch.where(h < 0.6, torch.zeros_like(h), h - 0.6)
    h.scatter_add_(1, torch.randint(0, GUIDE_BINS, (n_cells, 1), generator=g, device="cuda"),
                   torch.full((n_cells, 1), 4.0, device="cuda"))
    p = 0.9 * h.double() / h.double().sum(1, keepdim=True) + 0.1 / GUIDE_BINS
    cdf = torch.cumsum(p, 1)
    cdf[:, -1] = 1.0
    return cdf.float().cpu().numpy()


def _cache(case, scene, stream):
    kw = {}
    if case.get("octree"):
        kw = dict(octree=True, max_leaves=case["octree"], split_samples=4096.0 if case["octree"] > 4096 else 256.0)
    if case["tech"] & LIGHT:
        kw["arena_capacity"] = max(1 << 20, 2 * case["width"] * case["height"] * case["D"])
    return M.Cache(scene, case["grid"], case["tech"], case["D"], fp32_statistics=case.get("fp32", False),
                   stream=stream, **kw)


def prepare(case, seed):
    desc = _scene(case, seed)
    s = {"case": case, "seed": seed & 0x7FFFFFFF, "desc": desc, "stream": torch.cuda.Stream(), "it": 0}
    if case["kind"] == "first_image":
        desc.bvh = case["bvh"]
        return s
    st = s["stream"]
    s["scene"] = M.Scene(desc, stream=st)
    c = s["cache"] = _cache(case, s["scene"], st)
    s["image"] = torch.zeros(desc.n_pixels * 3, dtype=torch.float32, device="cuda")
    torch.cuda.synchronize()
    bd = bool(case["tech"] & LIGHT)
    if case["kind"] == "train":
        return s
    mode = case["mode"]
    # the job's first warm-up render; a bidirectional job's octree is refined by its sample counts
    c.render_iteration(s["image"], seed=s["seed"], iteration=0, mode=M.MARS_MODE_WARMUP, collect=bd,
                       vi_drop_brightest=10 if bd else 0, stream=st)
    if case["octree"]:
        c.update_counts(stream=st)
    if mode == "mars":
        q_rr, q_s, valid = _counts(case["scene"], c.n_cells, seed)
        est = _estimate(desc.width, desc.height, seed)
        kw = dict(guide_cdf=_guide(c.n_cells, seed)) if case["tech"] & GUIDED else {}
        c.set_state(q_rr=q_rr, q_s=q_s, valid=valid, pixel_estimate=est, run_sum=est * np.float32(N_ESTIMATE),
                    n_iterations=N_ESTIMATE, has_estimate=True, stream=st, **kw)
        if case["tune"]:
            c.autotune(seed=s["seed"], iteration=1, mode=M.MARS_MODE_MARS, repeats=1, stream=st)
    s["args"] = dict(seed=s["seed"], mode={"mars": M.MARS_MODE_MARS, "warmup": M.MARS_MODE_WARMUP,
                                           "fixed": M.MARS_MODE_FIXED}[mode],
                     weights=M.MARS_WEIGHTS_AWARE if case["aware"] else M.MARS_WEIGHTS_UNAWARE,
                     max_multiplicity=case["mult"], vi_drop_brightest=10 if bd else 0, combine=1 if bd else 0, stream=st)
    return s


_COUNTERS = ("rays", "vertices", "estimator_vertices", "light_rays", "connection_rays", "light_samples", "VI", "CI",
             "mean_beta")


def _outputs(image, stats):
    return {"image": image, **{k: stats[k] for k in _COUNTERS}}


def _full(a, n):
    out = np.zeros(n, a.dtype)
    out[:len(a)] = a
    return out


def run(s):
    case = s["case"]
    if case["kind"] == "first_image":
        st = s["stream"]
        scene = M.Scene(s["desc"], stream=st)
        cache = _cache(case, scene, st)
        image = np.empty(3 * cache.n_pixels, np.float32)
        stats = cache.render_iteration(image, seed=s["seed"], iteration=0, mode=M.MARS_MODE_WARMUP, max_multiplicity=16.0,
                                       stream=st)
        cache.close()
        scene.close()
        return _outputs(image, stats)
    c = s["cache"]
    it = s["it"] = (s["it"] + 1) % 65536
    if case["kind"] == "train":
        stats = c.render_iteration(s["image"], seed=s["seed"], iteration=it, mode=M.MARS_MODE_WARMUP, vi_drop_brightest=10,
                                   stream=s["stream"])
        c.update_counts(stream=s["stream"])
        g = c.get_state(stream=s["stream"])
        return {**_outputs(s["image"], stats), "q_rr": g["q_rr"], "q_s": g["q_s"], "valid": g["valid"],
                "run_sum": g["run_sum"], "pixel_estimate": g["pixel_estimate"], "oct_nodes": _full(g["oct_nodes"], c.oct_cap_nodes),
                "oct_leaf_level": _full(g["oct_leaf_level"], c.n_cells)}
    return _outputs(s["image"], c.render_iteration(s["image"], iteration=it, **s["args"]))


def work(case):
    """Operations and bytes of a pass whatever the implementation: the rays'
    traversals (two slab tests of 25 operations a node visit, about 45 a
    primitive test) and about 300 operations of sampling, evaluation and
    statistics a ray; the image, pixel estimate and running sum, the counts,
    statistics and guide tables and the scene, each moved once."""
    px = case["width"] * case["height"]
    fields, rays_px = FIELDS[case["scene"]]
    if case.get("mode", "warmup") != "mars":  # one continuation and one sample of each other technique per vertex
        rays_px = 1 + min(case["D"] - 1, {"box": 3, "room": 5}.get(case["scene"], 2)) * (3 if case["tech"] & LIGHT else 2)
    visits, tests = VISITS[case["scene"]]
    rays = px * rays_px
    cells = case["octree"] if case.get("octree") else case["grid"] ** 3
    n = case["prims"]
    prims = n + 16 if case["scene"] in ("box", "room") else 2 * n * n + 8 * n
    cell_bytes = 3 * (32 + 64) + (2048 if case["tech"] & GUIDED else 0)
    return {"bytes": px * (12 + 16 + 32) + cells * cell_bytes + prims * (64 + 64),
            "flops": rays * (50 * visits + 45 * tests + 300)}


def exact(case, seed):
    return None
