"""The per-tile lists at the sizes where the list sort changes its path: one warp or one CTA per
list, each number of keys a thread, lists cut into segments, segments that stay too large because
their primitives share a range, and rectangles counted and emitted by a whole warp, blocks split
over several warps.  Lists and records bit-exact against the oracle.  Marked gpu."""
import math

import numpy as np
import pytest
import torch

import oracle
from paper_2503_17491_gb300 import api, scenes
from gpu_common import check_lists, make_ctx, oracle_lists, to_dev

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _build():
    oracle.build()


def _one_tile(n, ranges, seed):
    """n primitives of about two columns' width in the directions of one tile's inner pixels, at
    the given ranges: each meets that tile and no other."""
    rng = np.random.default_rng(seed)
    g = math.pi - 2 * math.pi * (24 + rng.uniform(-4, 4, n)) / 64
    th = math.radians(10) * rng.uniform(-0.3, 0.3, n)
    p = np.stack([np.cos(th) * np.cos(g), np.cos(th) * np.sin(g), np.sin(th)], 1) * ranges[:, None]
    pl, q, ls = scenes.gaussians_on(p, -p, rng, jitter=0.0)
    ls[:] = np.log(0.04 * ranges)[:, None]
    view = scenes.View(np.eye(4), 16, 64, scenes.deg(-10), scenes.deg(10))
    return scenes.Scene(f"one_tile{n}", pl, q, ls, [view])


def _check(s, tile=(16, 16)):
    ctx = make_ctx(s.n, s.views, tile)
    ctx.render(*to_dev(s))
    assert ctx.status() == 0
    m = check_lists(ctx, s, s.views, tile)
    r = ctx.sorted_lists()[2].astype(np.int64)
    return m, int((r[:, 1] - r[:, 0]).max())


@pytest.mark.parametrize("n", [1, 31, 32, 33, 128, 129, 255, 256, 257, 1024, 1025, 2048, 2049,
                               4095, 4096, 4097, 8192, 20_001])
def test_list_lengths(n):
    rng = np.random.default_rng(n)
    assert _check(_one_tile(n, rng.uniform(2.0, 60.0, n), n))[1] == n


@pytest.mark.parametrize("n,kind", [(300, "equal"), (4096, "equal"), (9000, "equal"),
                                    (9000, "wall"), (20_000, "two")])
def test_shared_ranges(n, kind):
    """Ties are broken by the primitive id, and a bin of the segmentation that holds more than a
    segment's worth is merged: every primitive at one place, a thin wall behind a near object, and
    two places."""
    rng = np.random.default_rng(n)
    r = np.full(n, 7.0)
    if kind == "wall":
        r = 30.0 + 1e-4 * rng.uniform(0, 1, n)
        r[:5] = rng.uniform(0.5, 2.0, 5)
    s = _one_tile(n, r, 3)
    if kind != "wall":
        s.pos_logit[:, :3] = s.pos_logit[0, :3]
    if kind == "two":
        s.pos_logit[::2, :3] *= 1.5
    assert _check(s)[1] == n


@pytest.mark.parametrize("tile", [(16, 16), (8, 32), (32, 8), (4, 64)])
def test_wide_rectangles(tile):
    """Near, large primitives beside small ones: rectangles of one tile up to whole tile rows and
    every tile, across the seam, on a ragged image."""
    s = scenes.tiny_scene(700, 21, rows=45, cols=333, fov_deg=40, dist=(0.4, 6.0),
                          log_scale=(-3.0, 0.7))
    m, _ = _check(s, tile)
    assert m > 10 * s.n


@pytest.mark.parametrize("tile", [(16, 16), (8, 32), (32, 8), (4, 64)])
def test_split_blocks(tile):
    """A lone view whose blocks go to two and four warps against the same render with its blocks
    whole (a record pool too small for the split): images bit-identical, gradients equal up to the
    order of the float additions (each sum of k terms within k units of 2^-24 of its absolute
    terms; 1e-5 of the largest gradient covers the scene's sums)."""
    s = scenes.workload(1, n=30_000)
    v = s.views[0]
    dev = to_dev(s)
    ctx = make_ctx(s.n, [v], tile)
    a = ctx.render(*dev)
    st = ctx.stats()
    whole = api.SplatContext(s.n, 1, v.n_pixels, st["n_pairs"] + 8,
                             api.RenderConfig(tile_h=tile[0], tile_w=tile[1]),
                             max_tiles=st["n_tiles"])
    whole.set_views([v])
    b = whole.render(*dev)
    for x, y in zip(a, b):
        assert torch.equal(x, y)
    rng = np.random.default_rng(2)
    up = [torch.from_numpy(rng.normal(size=t.shape).astype(np.float32)).cuda() for t in a]
    ga, gb = ctx.backward(*dev, *up), whole.backward(*dev, *up)
    assert ctx.status() == 0 and whole.status() == 0
    for x, y in zip(ga, gb):
        assert (x - y).abs().max() <= 1e-5 * y.abs().max()


def _split_tiles(ctx):
    """Tiles whose blocks went to four and to two warps in the last render."""
    return ctx.debug_copy(6, 2, np.uint32).tolist()


@pytest.mark.parametrize("tile", [(16, 16), (8, 32), (32, 8), (4, 64)])
def test_split_levels(tile):
    """What decides on splitting, on both sides of each line.  The longest lists of two scans of a
    street are long against a warp's even share of the frame: their blocks go to four warps,
    others' to two, the shortest stay whole; images as with whole blocks (a record pool too small
    for the split), gradients equal up to the order of float additions (as in test_split_blocks).
    Over twelve such scans the same lists are below 2.65 shares, and nothing is split."""
    s = scenes.workload(1, n=60_000)
    v = s.views[0]
    dev = to_dev(s)
    warps = 3 * 8 * torch.cuda.get_device_properties(0).multi_processor_count

    def shares(ctx):   # entries of a block's list against an even share, longest first
        r = ctx.sorted_lists()[2].astype(np.int64)
        share = 8.0 * ctx.stats()["n_pairs"] / warps
        assert 0.4 * share > 64   # (shorter lists are never split)
        return np.sort(r[:, 1] - r[:, 0])[::-1] / share

    ctx = make_ctx(s.n, [v, v], tile)
    a = ctx.render(*dev)
    st = ctx.stats()
    sh = shares(ctx)
    n4, n2 = _split_tiles(ctx)
    assert sh[0] > 2.65 * 1.05 and n4 > 0 and n2 > 0 and n4 + n2 < len(sh)
    # lists go to four warps from 0.8 shares and to two from 0.4, both rounded up to a bucket of
    # list lengths, of which there are four an octave
    assert np.all(sh[:n4] >= 0.8) and np.all(sh[n4:n4 + n2] >= 0.4)
    assert np.all(sh[n4:] < 0.8 * 1.25) and np.all(sh[n4 + n2:] < 0.4 * 1.25)
    whole = api.SplatContext(s.n, 2, 2 * v.n_pixels, st["n_pairs"] + 8,
                             api.RenderConfig(tile_h=tile[0], tile_w=tile[1]),
                             max_tiles=st["n_tiles"])
    whole.set_views([v, v])
    b = whole.render(*dev)
    assert _split_tiles(whole) == [0, 0]
    assert all(torch.equal(x, y) for x, y in zip(a, b))
    up = [torch.ones_like(t) for t in a]
    for x, y in zip(ctx.backward(*dev, *up), whole.backward(*dev, *up)):
        assert (x - y).abs().max() <= 1e-5 * y.abs().max()
    many = make_ctx(s.n, [v] * 12, tile, max_pairs=16 * st["n_pairs"])
    many.render(*dev)
    assert shares(many)[0] < 2.65 * 0.95 and _split_tiles(many) == [0, 0]
    assert ctx.status() == 0 and whole.status() == 0 and many.status() == 0


def test_many_tiles():
    """A view of more tiles than the shared-memory counters hold (14,000), beside one of few: both
    in one call."""
    s = scenes.tiny_scene(3000, 5, rows=112, cols=32_000, dist=(0.6, 9.0), log_scale=(-5.0, -1.0))
    few = scenes.View(np.eye(4), 16, 64, scenes.deg(-20), scenes.deg(20))
    views = [s.views[0], few]
    ctx = make_ctx(s.n, views, (16, 16), max_pairs=1 << 21)
    ctx.render(*to_dev(s))
    assert ctx.status() == 0
    assert check_lists(ctx, s, views, (16, 16)) > s.n


def _rotation(rng):
    q = rng.normal(size=4)
    w, x, y, z = q / np.linalg.norm(q)
    return np.array([[1 - 2 * (y * y + z * z), 2 * (x * y - w * z), 2 * (x * z + w * y)],
                     [2 * (x * y + w * z), 1 - 2 * (x * x + z * z), 2 * (y * z - w * x)],
                     [2 * (x * z - w * y), 2 * (y * z + w * x), 1 - 2 * (x * x + y * y)]])


@pytest.mark.parametrize("kind", ["edge_on", "thin", "near", "far", "axes", "boundaries"])
@pytest.mark.parametrize("tile", [(16, 16), (4, 64)])
def test_boxes(kind, tile):
    """The projection's approximate box against the contract's where the bounds lie badly: planes
    seen edge on, slivers, primitives around and behind the sensor, far below a pixel, centres on
    the axes, poles and seam, and centres on pixel boundaries; from a level and two tilted poses,
    a narrow, a wide and a whole-sphere field of view."""
    rng = np.random.default_rng(len(kind) + tile[0])
    n = 6000
    g = rng.uniform(-math.pi, math.pi, n)
    th = np.arcsin(rng.uniform(-1, 1, n))
    r = np.exp(rng.uniform(math.log(0.05 if kind == "near" else 1.0),
                           math.log({"near": 1.5, "far": 400.0}.get(kind, 40.0)), n))
    if kind == "axes":
        g = rng.integers(-2, 3, n) * (math.pi / 2)
        th = rng.choice([0.0, 0.0, math.pi / 2, -math.pi / 2], n)
    if kind == "boundaries":
        g = math.pi - 2 * math.pi * rng.integers(0, 333, n) / 333
        th = math.radians(20) - math.radians(40) * rng.integers(0, 46, n) / 45
    p = np.stack([np.cos(th) * np.cos(g), np.cos(th) * np.sin(g), np.sin(th)], 1) * r[:, None]
    nrm = np.cross(p, rng.normal(size=(n, 3))) if kind == "edge_on" else rng.normal(size=(n, 3))
    pl, q, ls = scenes.gaussians_on(
        p, nrm, rng, jitter=0.0, quat_noise=0.0 if kind == "edge_on" else 0.05,
        log_scale=(-5.0, -2.5) if kind == "far" else (-3.5, -0.5))
    if kind == "thin":
        ls[:, 1] -= 6.0
    views = []
    for k, (rows, cols, fov) in enumerate([(45, 333, 20), (64, 128, 89), (33, 1000, 89.9)]):
        T = np.eye(4)
        if k:
            T[:3, :3] = _rotation(rng)
            T[:3, 3] = rng.normal(0, 0.3, 3)
        views.append(scenes.View(T, rows, cols, scenes.deg(-fov), scenes.deg(fov)))
    s = scenes.Scene(f"boxes_{kind}", pl, q, ls, views)
    ctx = make_ctx(s.n, views, tile, max_pairs=1 << 22)
    ctx.render(*to_dev(s))
    assert ctx.status() == 0
    assert check_lists(ctx, s, views, tile) > 0


@pytest.mark.parametrize("n,kind", [(70_000, "spread"), (65_536, "equal"), (70_000, "wall"),
                                    (70_001, "mixed"), (9000, "far"), (66_000, "far"),
                                    (30_000, "nested")])
def test_segments(n, kind):
    """Lists cut by one CTA and by a cluster, and segments that have to be cut again: all at one
    place (only the ids differ), a thin wall, a wall beside a spread, ranges past the last bin of
    the first cut, and clumps inside clumps that take several cuts."""
    rng = np.random.default_rng(n)
    r = rng.uniform(2.0, 60.0, n)
    if kind == "equal":
        r[:] = 7.0
    if kind == "wall":
        r = 30.0 + 1e-4 * rng.uniform(0, 1, n)
    if kind == "mixed":
        r[::3] = 12.0 + 1e-5 * rng.uniform(0, 1, len(r[::3]))
    if kind == "far":
        r = np.exp(rng.uniform(math.log(2.0 ** 21), math.log(2.0 ** 24), n))
    if kind == "nested":
        r = 16.0 + 8.0 * 2.0 ** -rng.integers(0, 22, n)
    s = _one_tile(n, r, 3)
    if kind == "equal":
        s.pos_logit[:, :3] = s.pos_logit[0, :3]
    assert _check(s)[1] == n


def _stage(s, name, runs=9, max_pairs=None):
    """Median time (ms) of a stage of a forward render."""
    ctx = make_ctx(s.n, s.views, max_pairs=max_pairs)
    dev = to_dev(s)
    ctx.set_profiling(True)
    ms = []
    for k in range(runs + 3):
        ctx.render(*dev)
        ms.append(ctx.stage_times()[name])
    assert ctx.status() == 0
    ctx.close()
    return float(np.median(ms[3:]))


def test_equal_ranges_cost_no_cliff():
    """150,000 primitives of one tile within a tenth of a millimetre of range are sorted in the
    order of time of as many spread over 60 m: they take one more cut (three more passes over the
    keys) and the same list sort.  Merging them in one CTA took 26 times as long."""
    rng = np.random.default_rng(1)
    n = 150_000
    wall = _stage(_one_tile(n, 30.0 + 1e-4 * rng.uniform(0, 1, n), 1), "tile sort")
    spread = _stage(_one_tile(n, rng.uniform(2.0, 60.0, n), 1), "tile sort")
    assert wall <= 5 * spread, (wall, spread)


def test_one_long_list_takes_several_ctas():
    """A list of 600,000 entries, cut by a cluster of CTAs, against one of 30,000 that one CTA cuts:
    twenty times the keys on four times the CTAs is five times as long, and the sort of the segments
    spreads over the SMs and adds less than that.  Cut by one CTA it took ten times as long."""
    rng = np.random.default_rng(2)
    t = {n: _stage(_one_tile(n, rng.uniform(2.0, 60.0, n), 1), "tile sort")
         for n in (30_000, 600_000)}
    assert t[600_000] <= 7 * t[30_000], t


def _wide_view(cols=32_000, rows=112):
    return scenes.View(np.eye(4), rows, cols, scenes.deg(-20), scenes.deg(20))


@pytest.mark.parametrize("tile", [(16, 16), (4, 64)])
@pytest.mark.parametrize("draws", [0, 2])
def test_bands(tile, draws):
    """Views counted in one band, in two and in several (the last band a single tile row), drawn or
    not: the lists of the drawn views against the oracle's."""
    s = scenes.tiny_scene(2500, 6, rows=16, cols=64, dist=(0.6, 9.0), log_scale=(-5.0, -1.0))
    views = [_wide_view(700, 45), _wide_view(), s.views[0], _wide_view(32_767, 225)]
    ctx = make_ctx(s.n, views, tile, max_pairs=1 << 22)
    if not draws:
        ctx.render(*to_dev(s))
        assert ctx.status() == 0
        check_lists(ctx, s, views, tile)
        return
    ctx.set_view_sampling(draws, 0.3, 5)
    seen = set()
    for _ in range(6):
        ctx.render(*to_dev(s))
        assert ctx.status() == 0
        on = ctx.active_views()
        seen.add(tuple(on))
        okeys, oids, _, _ = oracle_lists(s, views, tile)
        starts = np.cumsum([0] + [-(-v.rows // tile[0]) * -(-v.cols // tile[1]) for v in views])
        view = np.searchsorted(starts, (okeys >> np.uint64(32)).astype(np.int64), side="right") - 1
        gk, gv, _ = ctx.sorted_lists()
        np.testing.assert_array_equal(gk, (okeys >> np.uint64(32)).astype(np.uint32)[on[view]])
        np.testing.assert_array_equal(gv % s.n, oids[on[view]])
    assert len(seen) > 1


@pytest.mark.parametrize("wide", [False, True])
def test_lists_past_the_capacity(wide):
    """Lists keep the places below the capacity, each filled by a pair that belongs there, in
    order; the status says that pairs are missing."""
    s = scenes.tiny_scene(3000, 5, rows=112, cols=700, dist=(0.6, 9.0), log_scale=(-5.0, -1.0))
    views = [_wide_view() if wide else s.views[0]]
    ctx = make_ctx(s.n, views, max_pairs=1 << 21)
    ctx.render(*to_dev(s))
    assert ctx.status() == 0
    _, ids, ranges = ctx.sorted_lists()
    kappa = ctx.pair_records(s.n)["kappa"]
    cap = 2 * len(ids) // 3
    low = make_ctx(s.n, views, max_pairs=cap)
    low.render(*to_dev(s))
    assert low.status() == 1   # SPLAT_STATUS_CAPACITY
    _, got, cut = low.sorted_lists()
    assert len(got) == cap
    full = ranges[:, 1] > ranges[:, 0]
    np.testing.assert_array_equal(cut, np.where(full[:, None], np.minimum(ranges, cap), 0))
    for (a, b), (c, d) in zip(ranges[full].astype(np.int64), cut[full].astype(np.int64)):
        assert set(got[c:d]) <= set(ids[a:b]) and len(set(got[c:d])) == d - c
        key = list(zip(kappa[got[c:d]], got[c:d]))
        assert key == sorted(key)


def test_a_wide_view_costs_the_others_nothing():
    """Eleven views and one of more tiles than a CTA's counters hold are counted and emitted in one
    call in about the time of two calls (half as much again is allowed for the spread of times this
    short).  With a global atomic for every entry of every view it was 2.4 times."""
    s = scenes.workload(1, n=200_000)
    narrow = [scenes.View(s.views[0].T_ws, 64, 1024, scenes.deg(-22.5), scenes.deg(22.5))] * 11
    wide = [scenes.View(s.views[0].T_ws, 128, 32_000, scenes.deg(-22.5), scenes.deg(22.5))]
    ms = []
    for views in (narrow, wide, narrow + wide):
        s.views = views
        ms.append(_stage(s, "emission", max_pairs=1 << 24))
    assert ms[2] <= 1.5 * (ms[0] + ms[1]), ms


@pytest.mark.parametrize("n", [70_000, 600_000])
def test_clusters_under_capture(n):
    """A render whose list is cut by clusters, chained (up to 2^19 pairs) and not, replayed from a
    graph: the same images and lists as from plain launches."""
    rng = np.random.default_rng(n)
    s = _one_tile(n, rng.uniform(2.0, 60.0, n), 4)
    ctx = make_ctx(s.n, s.views)
    dev = to_dev(s)
    plain = [t.clone() for t in ctx.render(*dev)]
    lists = ctx.sorted_lists()
    out = ctx.alloc_images()
    graph = torch.cuda.CUDAGraph()
    torch.cuda.synchronize()
    with torch.cuda.graph(graph):
        ctx.render(*dev, out=out, stream=torch.cuda.current_stream())
    for _ in range(2):
        for t in out:
            t.zero_()
        graph.replay()
    torch.cuda.synchronize()
    assert ctx.status() == 0
    assert all(torch.equal(x, y) for x, y in zip(plain, out))
    for x, y in zip(lists, ctx.sorted_lists()):
        np.testing.assert_array_equal(x, y)
