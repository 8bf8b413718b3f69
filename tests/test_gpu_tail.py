"""The deep waves in two kernels (csrc/render.cu, k_tail and k_tail_reverse)
against the wave kernels: a profiled iteration renders with the wave kernels
alone, so the same iteration of the same state with and without `profile` gives
the same image and counters, and statistics that differ by the order of their
float additions only."""
import numpy as np
import pytest

import mars_workloads as W

pytestmark = pytest.mark.gpu

TECH3 = W.TECH_BSDF | W.TECH_NEE | W.TECH_GUIDED
KEYS = ("rays", "vertices", "estimator_vertices", "wave_entries", "shadow_entries", "shadow_traced", "wave_rays",
        "trace_work")


@pytest.fixture(scope="module")
def mars():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA GPU")
    from paper_2410_20429_gb300 import build as B
    B.build()
    import paper_2410_20429_gb300 as M
    return M


def _pair(mars, w, h, D, tech, lo, hi, cap=0, lanes=2):
    """(profiled, not profiled) results of one MARS iteration from the same state."""
    import torch
    sc = W.guided_room_scene(2, w, h, n_spheres=24)
    stream = torch.cuda.Stream()
    scene = mars.Scene(sc, stream=stream)
    c = mars.Cache(scene, 6, tech, D, arena_capacity=cap, lanes=lanes, stream=stream)
    q_rr, q_s, valid = W.random_count_fields(c.n_cells, seed=31, lo=lo, hi=hi)
    est = W.random_pixel_estimate(sc.n_pixels, seed=32, lo=0.2, hi=0.5)
    img = torch.zeros(3 * sc.n_pixels, dtype=torch.float32, device="cuda")
    out = []
    for profile in (True, False):
        st = dict(q_rr=q_rr, q_s=q_s, valid=valid, pixel_estimate=est, has_estimate=True, n_iterations=1,
                  stats=np.zeros((c.n_cells, 3, 8)))
        if tech & W.TECH_GUIDED:
            st.update(guide_hist=np.zeros((c.n_cells, 256), np.float32), guide_cdf=W.random_guide_cdf(c.n_cells, 33))
        c.set_state(stream=stream, **st)
        r = c.render_iteration(img, seed=6, iteration=3, mode=mars.MARS_MODE_MARS, profile=profile, stream=stream)
        torch.cuda.synchronize()
        out.append((img.cpu().numpy().copy(), r, c.get_state(stream=stream)))
    return out


def _same(a, b):
    (ia, ra, ga), (ib, rb, gb) = a, b
    assert np.array_equal(ia, ib)
    for k in KEYS:
        assert ra[k] == rb[k], k
    assert np.array_equal(ga["pixel_rays"], gb["pixel_rays"])
    np.testing.assert_allclose(ra["mean_beta"], rb["mean_beta"], rtol=1e-9)
    # float32 sums of runs of equal cells in a warp, in another grouping: 31 additions of 2^-24 each
    np.testing.assert_allclose(ga["stats"], gb["stats"], rtol=2e-6, atol=1e-9)
    if "guide_hist" in ga:
        np.testing.assert_allclose(ga["guide_hist"], gb["guide_hist"], rtol=1e-4, atol=1e-6)


# from the first wave on: pixel counts at the edges of a root group and of a block's
# rays, more pixels than the blocks' targets hold, every technique set and depth limit
@pytest.mark.parametrize("w,h,D,tech", [(1, 1, 10, TECH3), (7, 1, 3, TECH3), (8, 1, 3, 3), (9, 1, 4, 5), (131, 1, 2, TECH3),
                                        (64, 48, 1, 1), (97, 61, 10, TECH3), (256, 256, 5, 3), (255, 257, 4, TECH3)])
def test_whole_path_trees_equal_the_wave_kernels(mars, w, h, D, tech):
    a, b = _pair(mars, w, h, D, tech, 0.1, 0.6)
    assert a[1]["wave_launches"] == D and b[1]["wave_launches"] == 0
    _same(a, b)


# from a deeper wave on: images of more than 2^16 pixels, in one and two lanes
@pytest.mark.parametrize("w,h,lanes", [(300, 260, 1), (500, 300, 1), (500, 300, 2)])
def test_deep_waves_equal_the_wave_kernels(mars, w, h, lanes):
    a, b = _pair(mars, w, h, 8, TECH3, 0.05, 0.25, lanes=lanes)
    assert a[1]["wave_launches"] == 8 and 0 < b[1]["wave_launches"] < 8 * b[1]["tiles"]
    _same(a, b)


def test_slices_that_overflow_are_rendered_by_the_wave_kernels(mars):
    """A few pixels that split heavily in an arena whose average slice is ample:
    the tile is rendered again by the wave kernels and gives the same image."""
    import torch
    cfg = W.config_box(64, 64)
    q_rr, q_s, valid = W.random_count_fields(cfg.n_cells, seed=41, lo=0.2, hi=0.5)
    est = np.full((cfg.scene.n_pixels, 3), 0.5, np.float32)
    est[2000:2004] = 2e-3
    out = []
    for cap in (0, 45000):
        scene = mars.Scene(cfg.scene)
        c = mars.Cache(scene, cfg.grid_n, cfg.techniques, cfg.max_depth, arena_capacity=cap)
        c.set_state(q_rr=q_rr, q_s=q_s, valid=valid, pixel_estimate=est, has_estimate=True, n_iterations=1)
        img = torch.zeros(3 * cfg.scene.n_pixels, dtype=torch.float32, device="cuda")
        r = c.render_iteration(img, seed=2, iteration=1, mode=mars.MARS_MODE_MARS, profile=cap == 0)
        torch.cuda.synchronize()
        out.append((img.cpu().numpy().copy(), r, c.get_state()))
    assert out[1][1]["retries"] > 0
    assert np.array_equal(out[0][0], out[1][0]) and out[0][1]["rays"] == out[1][1]["rays"]
    np.testing.assert_allclose(out[0][2]["stats"], out[1][2]["stats"], rtol=2e-6, atol=1e-9)


# with light connections the small waves share launches of the shadow and light
# kernels: at every remainder of the batches and the depth limits of both techniques
@pytest.mark.parametrize("D", [1, 2, 3, 4, 5, 6, 7, 9])
def test_joined_side_kernels_equal_the_waves_own(mars, D):
    a, b = _pair(mars, 61, 47, D, W.TECH_BSDF | W.TECH_NEE | W.TECH_LIGHT, 0.3, 0.9)
    _same(a, b)
    assert b[1]["launches"] <= a[1]["launches"]
    for k in ("light_rays", "connection_rays", "light_samples"):
        assert a[1][k] == b[1][k], k


def test_a_tile_whose_slices_overflow_is_rendered_again_whole(mars):
    """The arena holds the tile with room to spare, but not the subtrees of a few
    pixels in their blocks' slices: one more attempt, of the same tile."""
    import torch
    cfg = W.config_box(64, 64)
    q_rr, q_s, valid = W.random_count_fields(cfg.n_cells, seed=41, lo=0.2, hi=0.5)
    est = np.full((cfg.scene.n_pixels, 3), 0.5, np.float32)
    est[2000:2004] = 2e-3
    scene = mars.Scene(cfg.scene)
    c = mars.Cache(scene, cfg.grid_n, cfg.techniques, cfg.max_depth, arena_capacity=45000)
    c.set_state(q_rr=q_rr, q_s=q_s, valid=valid, pixel_estimate=est, has_estimate=True, n_iterations=1)
    img = torch.zeros(3 * cfg.scene.n_pixels, dtype=torch.float32, device="cuda")
    r = c.render_iteration(img, seed=2, iteration=1, mode=mars.MARS_MODE_MARS)
    assert r["wave_entries"] < 45000
    assert r["retries"] == 1 and r["tiles"] == 2


@pytest.mark.parametrize("w,h,D", [(97, 61, 10), (300, 260, 8)])
def test_arena_demand_counts_every_depth(mars, w, h, D):
    """The rays the tile needed, whichever kernels rendered it (from the first
    wave on, from a deeper one on): all its depths' rays, so that an arena of that
    many slots holds the tile again."""
    a, b = _pair(mars, w, h, D, TECH3, 0.1, 0.6, lanes=1)
    assert a[1]["wave_launches"] > b[1]["wave_launches"]
    assert b[1]["arena_demand"] == a[1]["arena_demand"] == a[1]["wave_entries"]


def _box_job(mars, w, h, cap, lo, hi, est, lanes=1):
    """A MARS job of the box from given counts and a uniform pixel estimate: (cache, next iteration)."""
    import torch
    cfg = W.config_box(w, h)
    stream = torch.cuda.Stream()
    scene = mars.Scene(cfg.scene, stream=stream)
    c = mars.Cache(scene, cfg.grid_n, cfg.techniques, cfg.max_depth, arena_capacity=cap, lanes=lanes, stream=stream)
    q_rr, q_s, valid = W.random_count_fields(cfg.n_cells, seed=41, lo=lo, hi=hi)
    img = torch.zeros(3 * cfg.scene.n_pixels, dtype=torch.float32, device="cuda")
    c.set_state(q_rr=q_rr, q_s=q_s, valid=valid, pixel_estimate=np.full((cfg.scene.n_pixels, 3), est, np.float32),
                has_estimate=True, n_iterations=1, stream=stream)

    def step(it, **kw):
        kw = {"mode": mars.MARS_MODE_MARS, "update_estimate": False, **kw}
        r = c.render_iteration(img, seed=3, iteration=it, stream=stream, **kw)
        torch.cuda.synchronize()
        return r, img.cpu().numpy().copy()

    def estimate(e):
        c.set_state(pixel_estimate=e, has_estimate=True, n_iterations=1, stream=stream)
    return c, step, estimate


@pytest.mark.parametrize("cap", [400000, 280000])
def test_a_tile_the_arena_does_not_hold_is_split_at_once(mars, cap):
    """Counts that jump: the rays fill the arena, in k_tail or in a wave before it.
    The tile is split, without a second attempt as it is, into no more pieces than
    after the wave kernels' own attempt (whose estimate of the rays it lacks differs)."""
    out = []
    for profile in (True, False):
        c, step, estimate = _box_job(mars, 300, 260, cap, 0.05, 0.1, 0.5)
        step(1, profile=profile)
        estimate(np.full((c.n_pixels, 3), 0.01, np.float32))
        out.append(step(2, profile=profile))
    (a, ia), (b, ib) = out
    assert 1 < b["retries"] <= a["retries"] and b["tiles"] <= a["tiles"]
    assert np.array_equal(ia, ib) and a["rays"] == b["rays"]


def test_the_tail_comes_back_after_its_slices_overflowed(mars):
    """Three iterations whose few dear pixels overflow their blocks' slices, then even
    ones: k_tail renders whole path trees again."""
    c, step, estimate = _box_job(mars, 64, 64, 40000, 0.2, 0.5, 0.5)
    even = np.full((c.n_pixels, 3), 0.5, np.float32)
    dear = even.copy()
    dear[2000:2004] = 2e-3
    log = []
    for it in range(1, 160):
        if it <= 4:
            estimate(dear if it < 4 else even)
        log.append(step(it)[0])
    assert log[0]["retries"] > 0 and all(r["retries"] == 0 for r in log[4:])
    assert log[4]["wave_launches"] > 0 and log[-1]["wave_launches"] == 0


def test_nee_samples_that_overflow_their_slices_are_learned(mars):
    """Many more NEE samples than rays: one iteration finds out that the slices of the
    shadow region are too small, the next ones know."""
    import torch
    cfg = W.config_box(64, 64)
    stream = torch.cuda.Stream()
    scene = mars.Scene(cfg.scene, stream=stream)
    c = mars.Cache(scene, cfg.grid_n, cfg.techniques, cfg.max_depth, arena_capacity=30000, stream=stream)
    q = np.zeros((c.n_cells, 3, 3), np.float32)
    q[:, 0], q[:, 1] = 0.02, 1.0
    c.set_state(q_rr=q, q_s=0.9 * q, valid=np.ones((c.n_cells, 3), np.uint8), has_estimate=True, n_iterations=1,
                pixel_estimate=np.full((c.n_pixels, 3), 0.5, np.float32), stream=stream)
    log = [c.render_iteration(None, seed=2, iteration=it, mode=mars.MARS_MODE_MARS, update_estimate=False,
                              stream=stream) for it in range(1, 8)]
    assert log[0]["shadow_entries"] > 2 * log[0]["wave_entries"]
    assert all(r["retries"] == 0 for r in log[1:])


def test_a_steady_job_records_one_graph(mars):
    """An image of more than 2^16 pixels: the first iteration tells the depth of the
    tail, the next records the graph that all others replay."""
    c, step, _ = _box_job(mars, 300, 260, 0, 0.1, 0.3, 0.5)
    caps = []
    for it in range(6):
        step(it, mode=mars.MARS_MODE_WARMUP)
        caps.append(c.info()["graph_captures"])
    assert caps == [0, 1, 1, 1, 1, 1]


@pytest.mark.parametrize("w,h", [(310, 270), (480, 360)])
def test_a_job_that_alternates_records_each_graph_once(mars, w, h):
    """Fixed counts and learned ones in turn, whose waves call for two depths of the
    tail: the graph of each is recorded once."""
    c, step, _ = _box_job(mars, w, h, 0, 0.1, 0.3, 0.5)
    rays = [step(it, mode=(mars.MARS_MODE_FIXED, mars.MARS_MODE_MARS)[it & 1])[0]["wave_rays"][1] for it in range(12)]
    assert min(rays[::2]) > 65536 > max(rays[1::2])
    assert c.info()["graph_captures"] <= 2


def test_graphs_kept_are_few_and_replay_their_own_settings(mars):
    """Six settings in turn, more than are kept: each gives the image it gave at first."""
    c, step, _ = _box_job(mars, 64, 48, 0, 0.1, 0.3, 0.5)
    shapes = [([t] * 4, [0] * 4) for t in (32, 64, 96, 128, 160, 256)]
    first = None
    for it in range(3):
        for s in shapes:
            c.set_launch(*s)
            r, img = step(7, collect=False)
            first = img if first is None else first
            assert np.array_equal(img, first)
    assert c.info()["graph_captures"] == 18


def _both(mars, c, step):
    """An iteration by the wave kernels and by k_tail: images, counters and rays of every pixel the same."""
    out = []
    for profile in (True, False):
        r, img = step(profile)
        out.append((img, r, c.get_state()["pixel_rays"]))
    (ia, ra, pa), (ib, rb, pb) = out
    assert rb["wave_launches"] == 0 and np.array_equal(ia, ib) and np.array_equal(pa, pb)
    for k in KEYS:
        assert ra[k] == rb[k], k


FORMS = {"triangles": dict(tech=3), "guided_triangles": {}, "lbvh": {}, "many_spheres": {}, "warmup": dict(mode=0),
         "octree": dict(grid=4, cache=dict(octree=True, max_leaves=4096, split_samples=40.0)),
         "fixed": dict(mode=2), "unaware": dict(kw=dict(weights=1)), "fixed_unaware": dict(mode=2, kw=dict(weights=1)),
         "float32": dict(cache=dict(fp32_statistics=True)), "capped": dict(kw=dict(max_multiplicity=4.0))}


@pytest.mark.parametrize("form", FORMS)
def test_every_form_of_an_iteration_equals_the_wave_kernels(mars, form):
    import torch
    f = FORMS[form]
    tech = f.get("tech", TECH3)
    sc = W.guided_room_scene(2, 97, 61, n_spheres=900 if form == "many_spheres" else 24)
    if form in ("triangles", "guided_triangles", "lbvh"):
        sc = W.heightfield_scene(3, 40, 97, 61, n_spheres=30, n_lights=2, ggx_fraction=0.5)
        sc.bvh = int(form == "lbvh")
    scene = mars.Scene(sc)
    c = mars.Cache(scene, f.get("grid", 6), tech, 7, **f.get("cache", {}))
    img = torch.zeros(3 * sc.n_pixels, dtype=torch.float32, device="cuda")
    if form == "octree":
        c.render_iteration(img, seed=6, iteration=0, mode=mars.MARS_MODE_WARMUP)
        c.update_counts()
    q_rr, q_s, valid = W.random_count_fields(c.n_cells, seed=31, lo=0.1, hi=0.6)
    state = dict(q_rr=q_rr, q_s=q_s, valid=valid, has_estimate=True, n_iterations=1,
                 pixel_estimate=W.random_pixel_estimate(sc.n_pixels, seed=32, lo=0.2, hi=0.5))
    if tech & W.TECH_GUIDED:
        state["guide_cdf"] = W.random_guide_cdf(c.n_cells, 33)

    def step(profile):
        c.set_state(**state)
        r = c.render_iteration(img, seed=6, iteration=3, mode=f.get("mode", 1), profile=profile, **f.get("kw", {}))
        torch.cuda.synchronize()
        return r, img.cpu().numpy().copy()
    _both(mars, c, step)


def test_rays_at_the_edges_of_triangles_equal_the_wave_kernels(mars):
    """2.6 million camera rays and their second bounce over 131k triangles: one in some
    hundred thousand meets an edge to within the rounding of the edge functions, and
    which of two triangles it hits, or neither, is the same in both."""
    import torch
    sc = W.heightfield_scene(7, 256, 256, 256, n_spheres=64)
    scene = mars.Scene(sc)
    c = mars.Cache(scene, 8, 3, 3)
    img = torch.zeros(3 * sc.n_pixels, dtype=torch.float32, device="cuda")
    for it in range(40):
        def step(profile):
            r = c.render_iteration(img, seed=11, iteration=it, mode=mars.MARS_MODE_WARMUP, profile=profile)
            torch.cuda.synchronize()
            return r, img.cpu().numpy().copy()
        _both(mars, c, step)


@pytest.mark.parametrize("lanes", [1, 2])
@pytest.mark.parametrize("w", [440, 560, 700, 880])
def test_the_tail_starts_at_the_first_small_wave(mars, w, lanes):
    """At most 2^16 rays a lane and, where two lanes run at the same time, 3 * 2^14 a
    depth from there on over both.  The depth comes from the iteration before: waves
    of that many pixels differ from it by less than 5 %."""
    c, step, _ = _box_job(mars, w, 300, 0, 0.1, 0.3, 0.5, lanes=lanes)
    for it in range(2):
        r, _ = step(it, mode=mars.MARS_MODE_WARMUP)
    assert r["tiles"] == lanes and r["retries"] == 0
    waves, before = r["wave_rays"], r["wave_launches"] // r["tiles"]  # waves of the wave kernels
    load = [max(n / lanes / 65536, (lanes > 1) * np.mean(waves[k:]) / 49152) for k, n in enumerate(waves)]
    assert all(x > 0.95 for x in load[:before])
    assert before == len(waves) or load[before] < 1.05


@pytest.mark.parametrize("cap,threads,blocks", [(80000, 32, 1), (120000, 128, 2), (120000, 64, 4)])
def test_k_tail_keeps_to_the_room_a_launch_shape_leaves(mars, cap, threads, blocks):
    """Fewer blocks an SM than fit: k_tail has no more threads there than the wave
    kernels, seen by its slices, which are the larger the fewer blocks share the
    arena and then hold the subtrees of a few dear pixels."""
    out = []
    for shape in (None, ([threads] * 4, [blocks] * 4)):
        c, step, estimate = _box_job(mars, 64, 64, cap, 0.2, 0.5, 0.5)
        dear = np.full((c.n_pixels, 3), 0.5, np.float32)
        dear[2000:2004] = 2e-3
        estimate(dear)
        if shape:
            c.set_launch(*shape)
        out.append(step(1))
    (a, ia), (b, ib) = out
    assert a["retries"] == 1 and b["retries"] == 0 and b["wave_launches"] == 0
    assert np.array_equal(ia, ib) and a["rays"] == b["rays"]


def test_device_bytes_count_the_rounds_of_k_tail(mars):
    """A buffer of rounds (16 bytes each, 96 and one more a block) for every lane of a
    cache that may use k_tail."""
    scene = mars.Scene(W.guided_room_scene(2, 64, 64, n_spheres=24))
    for tech, has in ((TECH3, True), (W.TECH_BSDF | W.TECH_NEE | W.TECH_LIGHT, False)):
        one, two = (mars.Cache(scene, 6, tech, 5, lanes=n).info()["device_bytes"] for n in (1, 2))
        assert (two - one) % (16 * 97) == 0 and (two > one) == has


@pytest.mark.parametrize("D", [4, 5, 9])
def test_joined_side_kernels_are_fewer_launches(mars, D):
    """From four depths on the side kernels of several waves share launches."""
    a, b = _pair(mars, 61, 47, D, W.TECH_BSDF | W.TECH_NEE | W.TECH_LIGHT, 0.3, 0.9)
    assert b[1]["launches"] < a[1]["launches"]
