"""Traversal of the 4-wide hierarchy by pools of rays (csrc/render.cu) against
the oracle's brute-force hits: at the edges of a chunk of 32 rays, with the
grid's warps taking further chunks from the shared counter, and on a hierarchy
of many levels under both builders."""
import numpy as np
import pytest

import mars_workloads as W

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def mars():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA GPU")
    from paper_2410_20429_gb300 import build as B
    B.build()
    import paper_2410_20429_gb300 as M
    return M


def _lambert_room(w, h, nested):
    """The room with Lambertian spheres: values of a pixel then move with the
    rounding of a hit no more than the hit does (a glossy sphere amplifies it).
    nested: spheres that shrink by 0.7 towards one corner, a chain of a hierarchy."""
    sc = W.guided_room_scene(3, w, h, n_spheres=48)
    sc.materials[:, 0] = W.MAT_LAMBERT
    if nested:
        r = 1.6 * 0.7 ** np.arange(48)
        sc.spheres = np.stack([0.3 + r, 0.2 + r, 3.4 - r, 0.35 * r], 1).astype(np.float32).astype(np.float64)
    return sc


def _render(mars, sc, **kw):
    import torch
    s = mars.Scene(sc)
    c = mars.Cache(s, kw["grid_n"], kw["techniques"], kw["max_depth"])
    # one block of one warp per SM: waves larger than the grid's own rays use the shared counter
    c.set_launch([32] * 4, [1] * 4)
    img = torch.zeros(3 * sc.n_pixels, dtype=torch.float32, device="cuda")
    st = c.render_iteration(img, seed=4, iteration=0, mode=mars.MARS_MODE_WARMUP)
    return img.cpu().numpy().reshape(-1, 3).astype(np.float64), st


@pytest.mark.parametrize("w,h,bvh", [(1, 1, 0), (31, 1, 0), (33, 1, 1), (8, 8, 0), (97, 64, 0), (97, 64, 1)])
def test_closest_hits_of_camera_rays(mars, orc, w, h, bvh):
    """D = 1: a pixel is the radiance of the emitting quad its ray hits first, so
    each pixel tells which of 150 overlapping quads (each its own radiance, black
    from behind) was found.  At most one pixel in 500 may lie on an edge that
    float32 and float64 see differently (edges cover under 1e-5 of the image a
    float32 ulp wide; one pixel is allowed for each 500 started)."""
    rng = np.random.default_rng(8)
    n = 150
    p0, e1, e2 = rng.uniform(-2, 2, (n, 3)), rng.uniform(-1, 1, (n, 3)), rng.uniform(-1, 1, (n, 3))
    p0[:, 2] += 5
    away = np.einsum("ij,ij->i", np.cross(e1, e2), p0) > 0   # turn most of them to the camera
    away &= rng.uniform(size=n) < 0.8
    e1[away], e2[away] = e2[away], e1[away].copy()
    q = np.concatenate([p0, e1, e2], 1).astype(np.float32)
    sc = W.box_scene(w, h)
    sc.quads = q.astype(np.float64)
    sc.quad_mat = np.arange(n, dtype=np.int32)
    sc.materials = np.zeros((n, 8))
    sc.materials[:, 5:] = (1 + np.arange(n))[:, None] * np.array([1.0, 2.0, 4.0])
    sc.camera = np.array([0, 0, 0, 0, 0, 5, 0, 1, 0, 50.0])
    sc.bvh = bvh
    kw = dict(grid_n=4, techniques=W.TECH_BSDF, max_depth=1)
    g, _ = _render(mars, sc, **kw)
    o = orc.render(sc, iteration=0, seed=4, **kw)
    assert (g != o.image).any(axis=1).sum() <= -(-sc.n_pixels // 500) * (sc.n_pixels >= 500)


@pytest.mark.parametrize("w,h,bvh,nested", [(31, 1, 0, False), (33, 1, 1, False), (97, 64, 0, False), (97, 64, 0, True),
                                            (97, 64, 1, True)])
def test_hits_and_visibility_of_a_path_tree(mars, orc, w, h, bvh, nested):
    """Two bounces and their shadow rays: values within 1e-4 and rays alike for
    all but one pixel in 500 (a hit or a shadow edge seen differently)."""
    sc = _lambert_room(w, h, nested)
    sc.bvh = bvh
    kw = dict(grid_n=4, techniques=W.TECH_BSDF | W.TECH_NEE, max_depth=3)
    g, st = _render(mars, sc, **kw)
    o = orc.render(sc, iteration=0, seed=4, **kw)
    ok = (np.abs(g - o.image) <= 1e-4 * np.abs(o.image) + 1e-7).all(axis=1)
    assert (~ok).sum() <= -(-sc.n_pixels // 500) * (sc.n_pixels >= 500), np.flatnonzero(~ok)[:5]
    assert abs(st["rays"] - o.rays) <= 2e-3 * o.rays and abs(st["vertices"] - o.vertices) <= 2e-3 * o.vertices


@pytest.mark.parametrize("part,value", [((0, 1, 2), np.nan), ((0, 1, 2), np.inf), ((1,), -np.inf), ((0,), np.nan),
                                        ((3, 4, 5), np.nan), ((5,), np.inf)])
@pytest.mark.parametrize("w,h,lo,hi", [(33, 7, 0.1, 0.6), (97, 61, 0.1, 0.6)])
def test_rays_that_are_not_finite_meet_nothing(mars, w, h, lo, hi, part, value):
    """A camera whose origin (0..2) or look-at point (3..5) is not finite: every
    camera ray visits the root alone and misses."""
    import torch
    sc = _lambert_room(w, h, True)
    sc.camera = sc.camera.copy()
    sc.camera[list(part)] = value
    s = mars.Scene(sc)
    c = mars.Cache(s, 4, W.TECH_BSDF | W.TECH_NEE, 3)
    for profile in (True, False):
        img = torch.ones(3 * sc.n_pixels, dtype=torch.float32, device="cuda")
        st = c.render_iteration(img, seed=4, iteration=0, mode=mars.MARS_MODE_WARMUP, profile=profile)
        assert (img == 0).all() and st["rays"] == st["vertices"] == sc.n_pixels
        assert st["trace_work"] == [[2 * sc.n_pixels, 0, 0, 0], [0, 0, 0, 0]]
