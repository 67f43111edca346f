"""The traversal's dispatch at its edges: short and long queries, deep stacks,
frames small enough for a lane per sample, rays that are stopped.  Each is
compared, bit for bit, with the same work done another way by the library;
tests/test_gpu_tiny.py compares that with the oracle."""
import dataclasses

import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_2001_02620_gb300 import inputs as I

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def api():
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_2001_02620_gb300 import build as B
    B.build()
    from paper_2001_02620_gb300 import api as A
    return A


@pytest.fixture(scope="module")
def tiny(api):
    sc = I.tiny_scene()
    return sc, api.Scene(sc)


@pytest.fixture(scope="module")
def rays(tiny):
    lo, hi = I.scene_box(tiny[0])
    r = np.concatenate([I.rays_toward(150_000, lo - 30, hi + 30, I.instance_origins(tiny[0]), 1.5, seed=5),
                        I.rays_random(50_000, lo, hi, seed=6, tmax=60.0)])
    return torch.from_numpy(r[np.random.default_rng(7).permutation(len(r))]).cuda()


# warps of a full launch: 152 SMs x 32; its lanes 155,648
@pytest.mark.parametrize("n", [1, 31, 33, 1000, 4865, 60_000, 155_649])
@pytest.mark.parametrize("tuning", [dict(), dict(batch=3, block=64), dict(occupancy=48, fetch=16)])
def test_a_query_does_not_depend_on_its_company(tiny, rays, n, tuning):
    _, gs = tiny
    all_hits, all_bits = gs.trace_closest(rays), gs.trace_any(rays)
    hits, bits = gs.trace_closest(rays[:n], tuning=tuning), gs.trace_any(rays[:n], tuning=tuning)
    gs.check()
    assert torch.equal(hits, all_hits[:n])
    occ = (bits[:, None] >> torch.arange(32, device="cuda", dtype=torch.int32) & 1).reshape(-1)[:n]
    ref = (all_bits[:, None] >> torch.arange(32, device="cuda", dtype=torch.int32) & 1).reshape(-1)[:n]
    assert torch.equal(occ, ref)
    assert torch.equal(occ.bool(), hits[:, 1] != -1)  # the same interval: occluded means hit


def test_stacks_deeper_than_shared_memory(api):
    """A chain-shaped tree over coincident quads keeps three entries per level:
    64 of its quads stack some 60, four times what shared memory holds."""
    vv = np.array([[0, 0, 0], [1, 0, 0], [1, 1, 0], [0, 1, 0]], dtype=np.float32)
    q = np.tile(np.array([[0, 1, 2, 3]], dtype=np.uint32), (60, 1))
    sc = I.Scene([(vv, q)], I.IDENTITY_XFORM[None].copy(), np.zeros(1, dtype=np.uint32))
    rng = np.random.default_rng(3)
    o = np.concatenate([rng.uniform(-0.5, 1.5, size=(500, 2)), np.full((500, 1), 5.0)], 1)
    r = torch.from_numpy(I.ray_array(o, np.tile([[0.0, 0.0, -1.0]], (500, 1)))).cuda()
    deep, flat = api.Scene(sc, build_opts=dict(degenerate=1)), api.Scene(sc)
    for tuning in (dict(), dict(occupancy=48), dict(occupancy=16, fetch=16)):
        a, b = deep.trace_closest(r, tuning=tuning), deep.trace_any(r, tuning=tuning)
        deep.check()
        assert torch.equal(a, flat.trace_closest(r))
        assert torch.equal(b, flat.trace_any(r))
    assert (a[:, 1] != -1).sum() > 50


@pytest.mark.parametrize("quad", ["folded", "triangle"])
@pytest.mark.parametrize("side", [1.0, -1.0])
def test_retests_of_a_quad_by_the_triangles_it_hits(api, quad, side):
    """Rays along z on a grid over a quad (0,0,0) (1,0,0) (1,1,0) v3, its edges
    and diagonal included, which FP32 leaves to FP64.  Folded, v3 = (1,0,1): a
    ray with y <= x meets triangle 0 at z = 0 and triangle 1 at z = x - y.
    Triangle, v3 = v2: only triangle 0 has area.  All numbers are dyadic, so a
    re-test is exact; FP32 decisions are off by a few units in the last place
    of 5, and (u, v) are kept in 16 bits (half a step, 7.7e-6)."""
    v3 = [1, 0, 1] if quad == "folded" else [1, 1, 0]
    vv = np.array([[0, 0, 0], [1, 0, 0], [1, 1, 0], v3], dtype=np.float32)
    q = np.array([[0, 1, 2, 3]], dtype=np.uint32)
    gs = api.Scene(I.Scene([(vv, q)], I.IDENTITY_XFORM[None].copy(), np.zeros(1, dtype=np.uint32)))
    x, y = (a.ravel() for a in np.meshgrid(np.arange(-2, 19) / 16.0, np.arange(-2, 19) / 16.0))
    n = len(x)
    o = np.stack([x, y, np.full(n, 5.0 * side)], 1)
    r = I.ray_array(o, np.tile([[0.0, 0.0, -side]], (n, 1)))
    inside = (y >= 0) & (x <= 1) & (y <= x)
    only0 = quad == "triangle"
    far = 5.0 - side * (x - y)  # where triangle 1 is met, if it is there
    for skip in (False, True):  # skip: the interval starts beyond the nearer triangle
        near = np.full(n, 5.0) if only0 else np.minimum(5.0, far)
        other = np.full(n, np.inf) if only0 else np.maximum(5.0, far)
        ok = inside & (np.abs(x - y) >= 1 / 16) if skip else inside
        if skip:
            r[:, 3] = np.where(ok, near + 1 / 32, 0.0)
        t_ref = other if skip else near
        rt = torch.from_numpy(r).cuda()
        h = gs.trace_closest(rt).cpu().numpy()
        bits = gs.trace_any(rt).cpu().numpy()
        gs.check()
        hit = h[:, 1] != -1
        sel = ok if skip else np.ones(n, dtype=bool)
        want = ok & np.isfinite(t_ref)
        assert np.array_equal(hit[sel], want[sel])
        any_hit = (bits[:, None] >> np.arange(32) & 1).reshape(-1)[:n].astype(bool)
        assert np.array_equal(any_hit[sel], want[sel])
        w = want & sel
        t = h[:, 0].copy().view(np.float32)
        assert np.abs(t[w] - t_ref[w]).max(initial=0.0) <= 8 * 5 * 2.0**-23
        tri1 = (np.abs(t_ref - 5.0) > 1e-3) & (not only0)
        u, v = (h[:, 3] & 0xFFFF) / 65535.0, (h[:, 3] >> 16 & 0xFFFF) / 65535.0
        assert np.abs(u - np.where(tri1, y, x))[w].max(initial=0.0) <= 1e-5
        assert np.abs(v - np.where(tri1, x, y))[w].max(initial=0.0) <= 1e-5


def _views(sizes, spps):
    base, views = 0, []
    for (w, h), spp in zip(sizes, spps):
        views.append(dataclasses.replace(I.tiny_view(), w=w, h=h, spp=spp, pixel_base=base))
        base += w * h
    return views


@pytest.mark.parametrize("sizes,spps", [
    ([(1, 1)], [1]), ([(61, 47)], [1]), ([(5, 7)], [3]), ([(31, 33)], [8]), ([(31, 33)], [9]),
    ([(17, 3), (40, 21), (1, 1)], [2, 2, 2]), ([(17, 3), (40, 21)], [2, 3]), ([(192, 152)], [1]),
    ([(193, 152)], [1])])
def test_small_frames_equal_the_wavefront(api, tiny, sizes, spps):
    """Around the rule that takes small frames to the single kernel: images and
    path logs are those of the wavefront renderer."""
    sc, gs = tiny
    views = _views(sizes, spps)
    alb = torch.from_numpy(I.albedo(sc.n_quads)).cuda()
    params = I.Params(max_depth=4, sun_dir=I.MID_SUN_DIR, sun_E=(2.0, 2.0, 2.0), lights=I.tiny_lights())
    log = [torch.zeros(api.path_log_words(views, 4), dtype=torch.int32, device="cuda") for _ in range(2)]
    a = gs.render(views, alb, params, path_log=log[0])
    b = gs.render(views, alb, params, path_log=log[1], tuning=dict(mode=2))
    g = api.RenderGraph(gs, views, alb, params)
    c = g.launch()
    gs.check()
    for x, y, z in zip(a, b, c):
        assert torch.equal(x, y) and torch.equal(x, z)
    assert torch.equal(log[0], log[1])


@pytest.mark.parametrize("mode", [0, 1, 2])
def test_stopped_rays_are_reported_by_every_renderer(api, tiny, mode):
    sc, gs = tiny
    view = dataclasses.replace(I.tiny_view(), w=300, h=200)
    alb = torch.from_numpy(I.albedo(sc.n_quads)).cuda()
    gs.render([view], alb, I.tiny_params(), max_steps=3, tuning=dict(mode=mode))
    with pytest.raises(api.N.QrtError) as e:
        gs.check()
    assert e.value.code == api.N.QRT_ERR_STEP_LIMIT
    gs.check()  # cleared after reading


@pytest.mark.parametrize("tex", [False, True])
def test_adjoint_with_hits_kept_for_some_depths(api, tiny, tex):
    """The adjoint's replay follows the hits of its first pass for as many depths
    as the workspace has room for and traces the others: a workspace made by a
    render (no room) or by a shallower adjoint, which a captured call may not
    grow, gives the gradient of one with room for every depth."""
    sc, gs = tiny
    view = dataclasses.replace(I.tiny_view(), w=96, h=80, spp=3)
    alb = torch.from_numpy(I.albedo(sc.n_quads)).cuda()
    dimg = torch.from_numpy(np.random.default_rng(9).normal(size=(80, 96, 3)).astype(np.float32)).cuda()

    def params(depth):
        p = I.Params(max_depth=depth, sun_dir=I.MID_SUN_DIR, sun_E=(2.0, 2.0, 2.0), lights=I.tiny_lights())
        if tex:
            p.tex = torch.from_numpy(I.face_textures(sc.n_quads)).cuda()
        return p

    deep = params(4)
    ref = gs.adjoint([view], alb, [dimg], torch.zeros_like(alb), deep)
    gs.check()
    assert float(ref.abs().max()) > 0
    for before in (None, 2):
        s = torch.cuda.Stream()
        grad = torch.zeros_like(alb)
        with torch.cuda.stream(s):
            gs.render([view], alb, deep, tuning=dict(mode=2))
            if before:
                gs.adjoint([view], alb, [dimg], torch.zeros_like(alb), params(before))
            s.synchronize()
            g = torch.cuda.CUDAGraph()
            with torch.cuda.graph(g, stream=s):
                gs.adjoint([view], alb, [dimg], grad, deep)
            grad.zero_()
            g.replay()
        torch.cuda.synchronize()
        gs.check()
        # the same terms added by FP32 atomics in another order: at most a few
        # hundred terms to a quad, each rounded to 2^-24 of the sum of their sizes
        torch.testing.assert_close(grad, ref, rtol=1e-4, atol=1e-5 * float(ref.abs().max()))


def _nearly_coincident(copies, jitter):
    """The tiny scene with every instance `copies` times, a few units of FP32
    rounding apart: most rays have several nearest hits within their error
    bounds of each other."""
    sc = I.tiny_scene()
    x = np.repeat(sc.xforms, copies, axis=0).astype(np.float64)
    x += np.random.default_rng(1).uniform(-jitter, jitter, size=x.shape) * (np.abs(x) + 1.0)
    return I.Scene(sc.meshes, x.astype(np.float32), np.repeat(sc.mesh_ids, copies))


@pytest.mark.parametrize("copies,jitter", [(3, 1e-7), (4, 3e-7), (4, 1e-6)])
def test_near_ties_do_not_depend_on_the_company(api, copies, jitter):
    """A hit's bits, its distance included, are the same whatever other rays
    share the warp and whenever it gets to the FP64 tests."""
    sc = _nearly_coincident(copies, jitter)
    gs = api.Scene(sc)
    lo, hi = I.scene_box(sc)
    r = torch.from_numpy(I.rays_toward(300_000, lo - 30, hi + 30, I.instance_origins(sc), 1.5, seed=5)).cuda()
    ref = gs.trace_closest(r)
    for tuning in (dict(), dict(batch=8), dict(occupancy=32), dict(occupancy=32, block=64), dict(occupancy=24)):
        assert torch.equal(gs.trace_closest(r, tuning=tuning), ref)
    for seed in range(3):
        at = torch.randperm(len(r), device="cuda", generator=torch.Generator("cuda").manual_seed(seed))
        assert torch.equal(gs.trace_closest(r[at].contiguous()), ref[at])
    few = torch.cat([gs.trace_closest(r[k:k + 1].contiguous()) for k in range(3000)])
    gs.check()
    assert torch.equal(few, ref[:3000])


def test_captured_calls_outlive_larger_ones(api, tiny):
    """A render and an adjoint captured on a stream are replayed after calls that
    take more memory there: an adjoint of the same frame, a deeper one, one with
    textures, a larger frame."""
    sc, gs = tiny
    view = dataclasses.replace(I.tiny_view(), w=96, h=80, spp=3)
    alb = torch.from_numpy(I.albedo(sc.n_quads)).cuda()
    dimg = torch.from_numpy(np.random.default_rng(9).normal(size=(80, 96, 3)).astype(np.float32)).cuda()
    wave = dict(mode=2)

    def params(depth, tex=False):
        p = I.Params(max_depth=depth, sun_dir=I.MID_SUN_DIR, sun_E=(2.0, 2.0, 2.0), lights=I.tiny_lights())
        if tex:
            p.tex = torch.from_numpy(I.face_textures(sc.n_quads)).cuda()
        return p

    p2, p5, p5t = params(2), params(5), params(5, True)
    (ref,) = gs.render([view], alb, p5, tuning=wave)
    ref_grad = gs.adjoint([view], alb, [dimg], torch.zeros_like(alb), p2)
    torch.cuda.synchronize()
    s = torch.cuda.Stream()
    with torch.cuda.stream(s):
        out, grad, scratch = torch.zeros_like(ref), torch.zeros_like(alb), torch.zeros_like(alb)
        gs.render([view], alb, p5, outs=[out], tuning=wave)
        s.synchronize()
        g1, g2 = torch.cuda.CUDAGraph(), torch.cuda.CUDAGraph()
        with torch.cuda.graph(g1, stream=s):
            gs.render([view], alb, p5, outs=[out], tuning=wave)
        gs.adjoint([view], alb, [dimg], scratch, p2)
        s.synchronize()
        with torch.cuda.graph(g2, stream=s):
            gs.adjoint([view], alb, [dimg], grad, p2)
        more = [lambda: gs.adjoint([view], alb, [dimg], scratch, p5),
                lambda: gs.adjoint([view], alb, [dimg], scratch, p5t),
                lambda: gs.render([dataclasses.replace(view, w=400, h=300)], alb, p5, tuning=wave)]
        for call in more:
            call()
            out.zero_()
            grad.zero_()
            g1.replay()
            g2.replay()
            s.synchronize()
            assert torch.equal(out, ref)
            # the same terms, added by FP32 atomics in another order
            torch.testing.assert_close(grad, ref_grad, rtol=1e-4, atol=1e-5 * float(ref_grad.abs().max()))
    gs.check()


def test_two_shadow_rays_of_every_path_fit_their_queue(api):
    """A frame of exactly one chunk (2^13 paths) that looks straight down on a
    ground under a sun and a key light: every path queues two shadow rays, twice
    the paths of the chunk.  The cost map's own counters, which lie behind the
    queue, and the image stay what they are in sixteen chunks and in the
    single-kernel renderer."""
    rng = np.random.default_rng(4)
    c = rng.uniform(-20, 20, size=(300, 1, 3)) * [1, 1, 0] + [0, 0, 4]
    e = np.array([[-1, -1, 0], [1, -1, 0], [1, 1, 0], [-1, 1, 0]]) * rng.uniform(0.2, 0.8, size=(300, 1, 1))
    ground = np.array([[[-60, -60, 0], [60, -60, 0], [60, 60, 0], [-60, 60, 0]]])
    v = np.concatenate([c + e, ground]).astype(np.float32).reshape(-1, 3)
    sc = I.Scene([(v, np.arange(len(v), dtype=np.uint32).reshape(-1, 4))], I.IDENTITY_XFORM[None].copy(),
                 np.zeros(1, dtype=np.uint32))
    gs = api.Scene(sc)
    alb = torch.from_numpy(I.albedo(sc.n_quads)).cuda()
    view = I.View(eye=(0.0, 0.0, 50.0), look=(0.0, 0.0, 0.0), up=(0.0, 1.0, 0.0), vfov_deg=40.0, w=64, h=64, spp=2)
    light = np.array([[-5, -5, 30, 0, 10, 0, 10, 0, 0, 9, 8, 7]], dtype=np.float32)  # edge1 x edge2 points down
    params = I.Params(max_depth=2, sun_dir=(0.1, 0.2, 1.0), sun_E=(2.0, 2.0, 2.0), lights=light)
    n = 64 * 64 * 2
    maps, images = [], []
    for tuning in (dict(chunk_log2=13), dict(chunk_log2=10)):
        stats = torch.zeros(12, dtype=torch.int64, device="cuda")
        img = torch.empty((64, 64, 3), device="cuda")
        (cost,) = gs.cost_maps([view], alb, params, stats, outs=[img], tuning=tuning)
        gs.check()
        st = stats.cpu().numpy()
        assert st[6] == 2 * n and st[0] == 2 * n  # two shadow rays at depth 1; bounces leave upward or hit a quad's back
        assert int(torch.round(cost.double() * 2).sum()) == int(st[1] + st[7])
        maps.append(cost)
        images.append(img)
    (single,) = gs.render([view], alb, params, tuning=dict(mode=1))
    assert torch.equal(images[0], images[1]) and torch.equal(images[0], single)
    assert float((maps[0] - maps[1]).abs().mean()) <= 0.05 * float(maps[0].mean())


def _canopy(n, occluder_z=None):
    """Ground under n sheets parallel to the sun's direction (1, 0, 1), through
    whose overlapping boxes a shadow ray from the ground runs without a hit;
    optionally one quad across those rays, occluder_z above the ground.  Dyadic
    numbers: the sheets are exactly parallel to the rays."""
    rng = np.random.default_rng(1)
    c = np.stack([rng.uniform(-60, 36, n), rng.uniform(-20, 12, n), rng.uniform(20, 24, n)], 1)
    c = np.round(c * 64) / 64
    a, b = np.array([24.0, 0, 24]), np.array([0, 8.0, 0])
    q = np.stack([c, c + a, c + a + b, c + b], 1)
    if occluder_z is not None:
        p, u, w = np.array([occluder_z, 0, occluder_z]), np.array([3.0, 0, -3]), np.array([0, 3.0, 0])
        q = np.concatenate([q, np.stack([p - u - w, p + u - w, p + u + w, p - u + w])[None]])
    ground = np.array([[[-9, -9, 0], [9, -9, 0], [9, 9, 0], [-9, 9, 0]]])
    meshes = [(v.astype(np.float32).reshape(-1, 3), np.arange(4 * len(v), dtype=np.uint32).reshape(-1, 4))
              for v in (q, ground)]
    return I.Scene(meshes, np.stack([I.IDENTITY_XFORM] * 2), np.arange(2, dtype=np.uint32))


class _Limited:
    """Camera rays at the ground of a _canopy, shadow rays through its sheets."""

    def __init__(self, api, n, occluder_z=None):
        sc = _canopy(n, occluder_z)
        self.api, self.gs = api, api.Scene(sc)
        self.alb = torch.from_numpy(I.albedo(sc.n_quads)).cuda()
        self.params = I.Params(max_depth=1, sun_dir=(1.0, 0.0, 1.0), sun_E=(2.0, 2.0, 2.0))

    def view(self, side):
        return I.View(eye=(0.0, 0.0, 10.0), look=(0.0, 0.0, 0.0), up=(0.0, 1.0, 0.0), vfov_deg=20.0, w=side, h=side,
                      spp=1)

    def stopped(self, side, steps, mode):
        (img,) = self.gs.render([self.view(side)], self.alb, self.params, max_steps=steps, tuning=dict(mode=mode))
        try:
            self.gs.check()
        except self.api.N.QrtError as e:
            assert e.code == self.api.N.QRT_ERR_STEP_LIMIT
            return True, img
        return False, img

    def least(self, side):
        """The least limit that stops no ray of the single-kernel renderer, where
        each ray has one lane."""
        lo, hi = 1, 1 << 14
        while lo < hi:
            m = (lo + hi) // 2
            if self.stopped(side, m, 1)[0]:
                lo = m + 1
            else:
                hi = m
        return lo


@pytest.mark.parametrize("side", [1, 8])
def test_step_limit_of_shared_rays(api, side):
    """An unoccluded any-hit ray is stopped exactly where it is without help, and
    the lanes that help it stop with it: each of a warp's lanes makes at most the
    limit and a few turns more."""
    s = _Limited(api, 20_000)
    least = s.least(side)
    assert least > 500
    for mode in (1, 2):
        assert s.stopped(side, least - 1, mode)[0]
        assert not s.stopped(side, least, mode)[0]
    stats = torch.zeros(12, dtype=torch.int64, device="cuda")
    limit = 16
    for steps, most in ((0, side * side * least), (limit, side * side * 32 * (limit + 32))):
        if steps and least < 32 * (limit + 32) and side == 1:
            most = least // 2  # one ray alone: its helpers end far from the end of its tree
        stats.zero_()
        s.gs.render([s.view(side)], s.alb, s.params, max_steps=steps, tuning=dict(mode=2), stats=stats)
        if steps:
            with pytest.raises(api.N.QrtError):
                s.gs.check()
        else:
            s.gs.check()
        assert int(stats[7]) <= most


@pytest.mark.parametrize("z", [21.0, 23.0, 31.0, 45.0])
def test_an_answered_ray_is_not_charged_for_its_helpers(api, z):
    """An occluded ray that is answered within its limit without help is answered
    within it by a warp, whatever other lanes spend on the rest of its tree."""
    s = _Limited(api, 20_000, z)
    least = s.least(1)
    assert least > 200
    stopped, img = s.stopped(1, least, 2)
    assert not stopped
    assert torch.equal(img, s.stopped(1, 0, 1)[1])


def test_kept_hits_can_be_refused_and_are_given_back(api, tiny):
    """A large adjoint keeps its hits on the device (128 MiB here) until a call
    without them gives the memory back; the gradient is the same."""
    sc, gs = tiny
    view = dataclasses.replace(I.tiny_view(), w=512, h=512, spp=8)
    alb = torch.from_numpy(I.albedo(sc.n_quads)).cuda()
    dimg = torch.from_numpy(np.random.default_rng(9).normal(size=(512, 512, 3)).astype(np.float32)).cuda()
    p = I.Params(max_depth=4, sun_dir=I.MID_SUN_DIR, sun_E=(2.0, 2.0, 2.0))
    hits = 16 * 512 * 512 * 8 * 4
    s = torch.cuda.Stream()

    def grad(keep):
        g = torch.zeros_like(alb)
        gs.adjoint([view], alb, [dimg], g, p, keep_hits=keep)
        s.synchronize()
        return g, torch.cuda.mem_get_info()[0]

    with torch.cuda.stream(s):
        grad(False)  # the workspace
        without, free = grad(False)
        kept, less = grad(True)
        again, back = grad(False)
    gs.check()
    assert free - less >= hits // 2 and back - less >= hits // 2  # other allocations take and give a little
    # the same terms, added by FP32 atomics in another order
    tol = dict(rtol=1e-4, atol=1e-5 * float(kept.abs().max()))
    torch.testing.assert_close(without, kept, **tol)
    torch.testing.assert_close(again, kept, **tol)


def test_wavefront_splits_many_views(api, tiny):
    """More small views than one launch holds, by the wavefront (by default they
    take the single kernel), in one chunk and in several."""
    sc, gs = tiny
    views = _views([(16, 8 + k % 3) for k in range(70)], [1 + k % 2 for k in range(70)])
    alb = torch.from_numpy(I.albedo(sc.n_quads)).cuda()
    params = I.Params(max_depth=4, sun_dir=I.MID_SUN_DIR, sun_E=(2.0, 2.0, 2.0), lights=I.tiny_lights())
    whole = gs.render(views, alb, params, tuning=dict(mode=2))
    parts = gs.render(views, alb, params, tuning=dict(mode=2, chunk_log2=10))
    single = gs.render(views, alb, params, tuning=dict(mode=1))
    gs.check()
    for v, a, b, c in zip(views, whole, parts, single):
        assert torch.equal(a, b) and torch.equal(a, c)
    for k in (0, 63, 64, 69):
        assert torch.equal(gs.render([views[k]], alb, params, tuning=dict(mode=2))[0], whole[k])
