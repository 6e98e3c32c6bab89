"""Batches of jobs run as several launches or one, eagerly or as a captured
CUDA graph, through the C-ABI: with a fixed tile shape the images are
bit-identical to one launch over all views, and each scene's gradient is
the same sum over its views (up to float summation order)."""
from dataclasses import replace

import numpy as np
import pytest
import torch

from paper_2510_03312_gb300 import autotune as A
from paper_2510_03312_gb300 import raster
from paper_2510_03312_gb300 import scenes as S
from paper_2510_03312_gb300 import ubs as U

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_2510_03312_gb300 import build
    build.build()
    assert torch.cuda.is_available()


def _jobs():
    wl = S.workload_uneven_mix(seed=7, n_scenes=3, n_jobs=7, p_range=(2000, 20000), w_range=(40, 200),
                               h_range=(30, 160))
    ds = [raster.DeviceScene.from_scene(s) for s in wl.scenes]
    return wl, ds


def _reference(ds, views, cfg, dls_per_view):
    r = raster.Rasterizer(ds, views, cfg)
    r.forward(check=True)
    dL = torch.cat([d.reshape(-1) for d in dls_per_view])
    r.forward(check=False)
    g = [x.clone() for x in r.backward(dL)]
    imgs = [r.view_image(r.image, i).clone() for i in range(len(views))]
    return imgs, g


def _dl_per_view(views, seed=0):
    rng = np.random.default_rng(seed)
    return [torch.from_numpy(rng.uniform(-1, 1, (3, v.height, v.width)).astype(np.float32)).cuda() * 1e-3
            for v in views]


def _batch_dls(b, per_view):
    out = b.dL_like()
    for gi, g in enumerate(b.groups):
        r = b.rasterizers[gi]
        for k, i in enumerate(g):
            r.view_image(out[gi], k).copy_(per_view[i])
    return out


def _close(a, b, rel=1e-5):
    scale = max(float(b.abs().max()), 1e-12)
    return float((a - b).abs().max()) <= rel * scale


@pytest.mark.parametrize("name", list(A.SCHEDULES))
@pytest.mark.parametrize("graph", [False, True])
def test_batch_schedules_match_one_launch(name, graph):
    wl, ds = _jobs()
    per_view = _dl_per_view(wl.views)
    ref_img, ref_g = _reference(ds, wl.views, wl.cfg, per_view)
    b = raster.Batch(ds, wl.views, wl.cfg, A.SCHEDULES[name](wl.scenes, wl.views))
    b.size()
    dls = _batch_dls(b, per_view)
    if graph:
        g = b.capture(dls)
        for x in b.grads:
            x.fill_(123.0)  # a replay must re-zero and rebuild them
        g.replay()
    else:
        b.step(dls)
    torch.cuda.synchronize()
    assert all(st.status == 0 for st in b.status())
    for i in range(len(wl.views)):
        assert torch.equal(b.image(i), ref_img[i]), f"view {i} differs"
    for s, (x, y) in enumerate(zip(b.grads, ref_g)):
        assert _close(x, y), f"scene {s}: {float((x - y).abs().max()):.3e}"


@pytest.mark.parametrize("tile", A.TILES)
def test_batch_tile_shapes_agree(tile):
    wl, ds = _jobs()
    per_view = _dl_per_view(wl.views)
    ref_img, ref_g = _reference(ds, wl.views, wl.cfg, per_view)
    cfg = replace(wl.cfg, tile_w=tile[0], tile_h=tile[1])
    b = raster.Batch(ds, wl.views, cfg, A.one_launch(wl.scenes, wl.views))
    b.size()
    b.step(_batch_dls(b, per_view))
    torch.cuda.synchronize()
    for i in range(len(wl.views)):
        # the tile origin enters the staged mean's rounding: 1e-4 is the image bound
        assert float((b.image(i) - ref_img[i]).abs().max()) <= 1e-4
    for x, y in zip(b.grads, ref_g):
        assert _close(x, y, rel=1e-3)


def test_device_autotune_returns_a_valid_plan():
    wl, ds = _jobs()
    meas = A.device_measure(ds, wl.views, wl.cfg, steps=2, warmup=1)
    plan = A.tune(wl.scenes, wl.views, wl.cfg, meas, tiles=((16, 16), (32, 32)),
                  schedules={k: A.SCHEDULES[k] for k in ("one_launch", "per_view")})
    assert plan.tile in ((16, 16), (32, 32)) and plan.ms > 0
    assert len(plan.table) == 4 * len(A.FORMS)


@pytest.mark.parametrize("form", ["persistent", "split"])
@pytest.mark.parametrize("tile", A.TILES)
@pytest.mark.parametrize("graph", [False, True])
def test_launch_forms_match_the_grid(form, tile, graph):
    """The persistent launch form of both blend kernels, and the split-list
    form on lists that need no split, give the grid form's images bit for
    bit and the same gradients (up to float summation order), on three
    steps in a row (the persistent tile counters and the split plan's
    counters reset themselves), eagerly and replayed from a captured graph."""
    wl, ds = _jobs()
    cfg = replace(wl.cfg, tile_w=tile[0], tile_h=tile[1])
    per_view = _dl_per_view(wl.views)
    ref_img, ref_g = _reference(ds, wl.views, cfg, per_view)
    b = raster.Batch(ds, wl.views, replace(cfg, **A.form_fields(form)), A.one_launch(wl.scenes, wl.views))
    b.size()
    dls = _batch_dls(b, per_view)
    graph_obj = b.capture(dls) if graph else None
    for step in range(3):
        if graph:
            graph_obj.replay()
        else:
            b.step(dls)
        torch.cuda.synchronize()
        assert all(st.status == 0 for st in b.status())
        for i in range(len(wl.views)):
            assert torch.equal(b.image(i), ref_img[i]), f"step {step}: view {i} differs"
        for s, (x, y) in enumerate(zip(b.grads, ref_g)):
            assert _close(x, y), f"step {step}, scene {s}: {float((x - y).abs().max()):.3e}"


def test_dense_lists_over_many_tiles_match_views_alone():
    """Three 1600x1060 views of the 1M-primitive scene in one launch (20,100
    tiles, about 250 instances a tile): the blend kernels take the tiles
    longest list first, through the multi-block ordering, and every image is
    bit-identical to its view rendered alone (6,700 tiles, ordered by one
    block) and the gradient is the sum of the views' gradients."""
    rng = np.random.default_rng(5)
    sc = S.make_scene(1, 3, 1_000_000, means="clusters", extent=5.0, rng=rng)
    views = S.sphere_views(rng, 3, 8.0, 1600, 1060)
    cfg = S.RasterConfig()
    ds = [raster.DeviceScene.from_scene(sc)]
    per_view = _dl_per_view(views, seed=3)
    r = raster.Rasterizer(ds, views, cfg)
    r.forward(check=True)
    NT = r.n_tiles()
    st = r.status()
    assert NT > 16384 and st.instances >= 64 * NT and r.capacity >= 64 * NT
    r.forward(check=False)
    g = r.backward(torch.cat([d.reshape(-1) for d in per_view]))[0].clone()
    g_sum = torch.zeros_like(g)
    for i, v in enumerate(views):
        r1 = raster.Rasterizer(ds, [v], cfg)
        r1.forward(check=True)
        assert r1.status().instances >= 64 * r1.n_tiles()
        img1 = r1.forward(check=False)
        assert torch.equal(r.view_image(r.image, i), r1.view_image(img1, 0)), f"view {i} differs"
        g_sum += r1.backward(per_view[i].reshape(-1))[0]
        del r1
    assert _close(g, g_sum)
    # the persistent form takes the same longest-first order from its counter
    rp = raster.Rasterizer(ds, views, replace(cfg, persistent=True))
    rp.forward(check=True)
    for _ in range(2):
        imgp = rp.forward(check=False)
        gp = rp.backward(torch.cat([d.reshape(-1) for d in per_view]))[0]
        torch.cuda.synchronize()
        assert torch.equal(imgp, r.image)
        assert _close(gp, g)


@pytest.mark.parametrize("tile", [(8, 8), (16, 16), (16, 32), (32, 32)])
@pytest.mark.parametrize("n,cap", [(2049, None), (2304, None), (9000, None), (9000, 3_000_000)])
def test_split_segments_at_their_edges(tile, n, cap):
    """One tile's list one entry over the split length, at a multiple of the
    shortest segment and many segments long, with a workspace that holds the
    shortest segments and (a capacity far above the lists) one that holds
    fewer, per tile shape: the image within 1e-5 of the unsplit form's and
    the gradients within 1e-3 of their plane's largest, the bounds of the
    oracle comparisons."""
    rng = np.random.default_rng(n)
    sc = S.make_scene(n, 3, n, scale_range=(0.02, 0.05), rng=rng)
    sc.plane("mean_x")[:] = (0.0005 * rng.uniform(-1.0, 1.0, (3, n))).astype(np.float32)
    # the shorter lists' pixel stays above T_min to their end, the long one's ends in some middle segment
    op = rng.choice([0.0043, 0.01], n, p=[0.98, 0.02]) if n < 9000 else rng.choice([0.005, 0.02, 0.1], n)
    sc.plane("opacity")[:] = op.astype(np.float32)
    v = S.make_view(np.eye(3), np.array([0.0, 0.0, 4.0]), 75, 71)  # the stack's mean at a pixel's centre
    got = {}
    for split in (False, True):
        r = raster.Rasterizer([raster.DeviceScene.from_scene(sc, device="cuda")], [v],
                              S.RasterConfig(tile_w=tile[0], tile_h=tile[1], split_lists=split), capacity=cap,
                              device="cuda")
        for _ in range(2):  # the second on the segment state the first left
            r.preprocess()
            r.bin_sort()
            img = r.render_fwd().clone()
        st = r.status()
        assert st.status == 0 and torch.diff(r.export(U.EXPORT_TILE_START)).max() > 2048
        dL = torch.sin(torch.arange(img.numel(), device="cuda")) / img.numel()
        got[split] = img, r.backward(dL)[0].clone()
    assert (got[True][0] - got[False][0]).abs().max() <= 1e-5
    worst = ((got[True][1] - got[False][1]).abs().amax(1) / got[False][1].abs().amax(1).clamp(min=1e-30)).max()
    assert worst <= 1e-3, float(worst)


@pytest.mark.parametrize("n", [4096, 4097, 8192, 8193, 20000])
def test_long_lists_joined_by_rank(n):
    """Lists at and around the 4096 entries of one sorted segment, in the
    split form (segments sorted by separate CTAs and joined by rank) and the
    other (merged by one CTA): the same lists, bit for bit, and in the order of
    (depth, record); with many records at one depth."""
    rng = np.random.default_rng(n)
    sc = S.make_scene(n, 3, n, scale_range=(0.02, 0.05), rng=rng)
    sc.plane("mean_x")[:] = (0.0005 * rng.uniform(-1.0, 1.0, (3, n))).astype(np.float32)
    sc.plane("mean_x")[2] = rng.choice(np.linspace(-0.5, 0.5, 97).astype(np.float32), n)
    v = S.make_view(np.eye(3), np.array([0.0, 0.0, 4.0]), 75, 71)
    lists = []
    for split in (False, True):
        r = raster.Rasterizer([raster.DeviceScene.from_scene(sc, device="cuda")], [v], S.RasterConfig(split_lists=split),
                              device="cuda")
        r.forward(check=True)
        k = int(r.status().instances)
        lists.append((r.export(U.EXPORT_TILE_START).clone(), r.export(U.EXPORT_INSTANCES)[:k].clone()))
        keys = r.export(U.EXPORT_KEYS).cpu().numpy().view(np.uint32)
    assert all(torch.equal(a, b) for a, b in zip(*lists))
    start, inst = (t.cpu().numpy().view(np.uint32).astype(np.int64) for t in lists[1])
    assert np.diff(start).max() >= 4096
    for s, e in zip(start[:-1], start[1:]):
        order = inst[s:e]
        assert np.array_equal(order, order[np.lexsort((order, keys[order]))]) and np.unique(order).size == order.size


@pytest.mark.parametrize("tile", [(8, 8), (16, 16), (16, 32), (32, 32)])
def test_few_tiles_match_many(tile):
    """A view alone (few tiles: the forward that evaluates four entries ahead)
    and the same view among enough copies to fill the GPU (the general form):
    images, final T and last contributors bit for bit."""
    rng = np.random.default_rng(tile[0] + tile[1])
    sc = S.make_scene(9, 3, 3001, scale_range=(0.02, 0.2), rng=rng)
    v = S.make_view(np.eye(3), np.array([0.0, 0.0, 3.0]), 101, 77)
    tiles = -(-v.width // tile[0]) * -(-v.height // tile[1])
    warps = tiles * tile[0] * tile[1] // 64
    n = 152 * 4 * 2 // warps + 1
    assert warps <= 152 * 4 * 2 < n * warps and n <= 256
    got = []
    for k in (1, n):
        r = raster.Rasterizer([raster.DeviceScene.from_scene(sc, device="cuda")], [v] * k,
                              S.RasterConfig(tile_w=tile[0], tile_h=tile[1]), device="cuda")
        r.forward(check=True)
        px = v.width * v.height
        got.append((r.image[:3 * px].clone(), r.export(U.EXPORT_FINAL_T)[:px].clone(), r.export(U.EXPORT_LAST)[:px].clone()))
    assert all(torch.equal(a, b) for a, b in zip(*got))


def _planned_segment(r, lists):
    """Entries per segment that the split form plans for these list lengths
    (uint32 per tile), restated from the rule: the shortest of 128 (or the
    blend's batch of 256 entries for tiles over 256 pixels) and its doublings
    up to 2048 of which there are at most 16 per SM and whose state the
    workspace holds."""
    def up(x):
        return (x + 255) // 256 * 256
    px = int(r.cfg.tile_w) * int(r.cfg.tile_h)
    nt, cap = r.n_tiles(), r.capacity
    ms = cap // 2048 + 1
    aside = up(16 * ms) + up(4 * nt) + up(2 * ms * px * 32) + up(8 * ms) + 2 * up(4 * ms)
    room = up(8 * r.n_pix) + aside - up(16 * ms) - up(4 * nt) - up(4 * ms * px) - up(4 * ms)
    slots = min((room - 1024) // (20 * px + 8), cap // 128 + ms)
    safe = 128
    while safe < 2048 and cap // safe + ms > slots:
        safe *= 2
    chunks = int(sum(-(-int(n) // 512) for n in lists if n > 512))
    length = 128 if px <= 256 else 256
    while length < 2048 and (chunks * 512 > 152 * 16 * length or
                             (length < safe and chunks * max(1, 512 // length) > slots)):
        length *= 2
    return length


def _used_segment(r, lists):
    """Entries per segment that the kernels used: the split tiles' table
    (tile, first slot, segments, first extra segment) found in the workspace
    by its tiles."""
    tiles = np.flatnonzero(lists > 2048)
    off = r.ws_ptr - r._ws.data_ptr()
    words = r._ws[off:off + r.ws_bytes // 4 * 4].cpu().numpy().view(np.uint32)
    found = set()
    for o in range(0, words.size - 4 * tiles.size, 64):  # on 256-byte boundaries
        if words[o] not in tiles:
            continue
        t = words[o:o + 4 * tiles.size].reshape(-1, 4)
        if not np.array_equal(np.sort(t[:, 0]), tiles):
            continue
        for length in (128, 256, 512, 1024, 2048):
            if np.array_equal(t[:, 2], -(-lists[t[:, 0]].astype(np.int64) // length)):
                found.add(length)
    assert len(found) == 1, found
    return found.pop()


def _split_against_unsplit(sc, view, tile, capacity):
    """Renders in both forms: the images within 1e-5, the gradients within 1e-3
    of their plane's largest and the lists bit for bit; returns the split
    form's rasterizer and its list lengths."""
    got = {}
    for split in (False, True):
        r = raster.Rasterizer([raster.DeviceScene.from_scene(sc, device="cuda")], [view],
                              S.RasterConfig(tile_w=tile[0], tile_h=tile[1], split_lists=split),
                              capacity=capacity, device="cuda")
        for _ in range(2):  # the second on the segment state the first left
            r.preprocess()
            r.bin_sort()
            img = r.render_fwd().clone()
        st = r.status()
        assert st.status == 0
        start = r.export(U.EXPORT_TILE_START).clone()
        inst = r.export(U.EXPORT_INSTANCES)[:int(st.instances)].clone()
        lists = torch.diff(start).cpu().numpy().astype(np.uint32)
        length = (_planned_segment(r, lists), _used_segment(r, lists)) if split else None
        dL = torch.sin(torch.arange(img.numel(), device="cuda")) / img.numel()
        got[split] = img, r.backward(dL)[0].clone(), start, inst
    assert torch.equal(got[True][2], got[False][2]) and torch.equal(got[True][3], got[False][3])
    assert (got[True][0] - got[False][0]).abs().max() <= 1e-5
    worst = ((got[True][1] - got[False][1]).abs().amax(1) / got[False][1].abs().amax(1).clamp(min=1e-30)).max()
    assert worst <= 1e-3, float(worst)
    assert length[0] == length[1], length
    return length[1], lists


@pytest.mark.parametrize("tile,length", [((8, 8), 256), ((16, 16), 512), ((16, 32), 512), ((32, 32), 1024)])
def test_split_segments_of_a_tight_workspace(tile, length):
    """One long list and a capacity that just holds it: the workspace has state
    for few segments, and they are longer than the shortest."""
    n = 9000
    rng = np.random.default_rng(n)
    sc = S.make_scene(n, 3, n, scale_range=(0.001, 0.002), rng=rng)
    sc.plane("mean_x")[:] = (0.0005 * rng.uniform(-1.0, 1.0, (3, n))).astype(np.float32)
    sc.plane("opacity")[:] = rng.choice([0.005, 0.02, 0.1], n).astype(np.float32)
    v = S.make_view(np.eye(3), np.array([0.0, 0.0, 4.0]), 75, 71)  # the stack's mean in one tile, whatever its shape
    used, lists = _split_against_unsplit(sc, v, tile, capacity=n)
    assert used == length and lists.max() == n == lists.sum()


@pytest.mark.parametrize("n,size,length,joined", [(4500, (96, 64), 256, True), (20000, (64, 48), 512, True),
                                                  (8000, (128, 96), 1024, False), (20000, (96, 64), 1024, False)])
def test_split_segments_of_many_long_lists(n, size, length, joined):
    """Every tile's list is long: more entries than segments of the shortest
    length may number, so that they are longer though the workspace has state
    for more, and lists over 4096 entries joined by rank up to 2048 chunks of
    512 and merged in rounds beyond."""
    rng = np.random.default_rng(n)
    sc = S.make_scene(n, 3, n, scale_range=(8.0, 12.0), rng=rng)
    sc.plane("mean_x")[:] = rng.uniform(-0.3, 0.3, (3, n)).astype(np.float32)
    sc.plane("opacity")[:] = rng.choice([0.006, 0.02], n, p=[0.97, 0.03]).astype(np.float32)
    v = S.make_view(np.eye(3), np.array([0.0, 0.0, 4.0]), *size)
    used, lists = _split_against_unsplit(sc, v, (8, 8), capacity=3_000_000)
    assert used == length and (lists > 2048).all() and lists.max() > 4096
    chunks = int((-(-lists.astype(np.int64) // 512)).sum())
    assert (chunks <= 2048) == joined, chunks
