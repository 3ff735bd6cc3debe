"""The radix sorts of the split sort at the sizes where their tiles, look-back
groups and launch shapes change: the depth order of the points and the
(tile, depth, index) order of the copies against NumPy's stable sorts of the
same integer keys. Exact: the keys are integers, so no tolerance."""
import numpy as np
import pytest
import torch

from paper_2508_19140_gb300 import scenes

from gpu_util import Run

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _need_gpu():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2508_19140_gb300 import build
    build.build()


def _view(n, width, height, depths, seed):
    rng = np.random.default_rng(seed)
    f = 0.9 * width
    z = {"spread": rng.uniform(0.5, 60.0, n), "equal": np.full(n, 3.0), "two": rng.choice([2.0, 5.0], n),
         "culled": np.where(rng.random(n) < 0.7, -1.0, rng.uniform(1.0, 2.0, n))}[depths]
    xyz = np.stack([rng.uniform(-0.6, 0.6, n) * width / f * z, rng.uniform(-0.6, 0.6, n) * height / f * z, z], 1)
    return scenes.View(xyz=xyz.astype(np.float32), opacity=rng.random(n).astype(np.float32),
                       feat=rng.random((n, 1)).astype(np.float32), camera=scenes.identity_camera(width, height, f))


def _bits(x):
    return np.asarray(x, np.float32).view(np.uint32).astype(np.int64)


def _check(views, tile=16):
    r = Run(views, tile=tile)
    assert r.status == 0
    n = sum(len(v.xyz) for v in views)
    zb = r.arr("zbits", np.uint32, n).astype(np.int64)
    p4 = r.arr("rect", np.uint32, n).astype(np.int64)
    image = np.repeat(np.arange(len(views)), [len(v.xyz) for v in views])
    cull = int(_bits(views[0].camera.far))
    # (image, depth bits, index): culled points behind every visible one of their image
    depth = np.lexsort((np.arange(n), np.where(p4 == 0xFFFFFFFF, cull, zb), image))
    assert np.array_equal(r.arr("depth_sorted", np.uint32, n), depth.astype(np.uint32))
    _check_copies(r, views, tile, depth, image, (p4 & 0xFFFF, (p4 >> 16) & 0x3FFF, (p4 >> 30) & 1, p4 >> 31),
                  p4 != 0xFFFFFFFF)


def _check_copies(r, views, tile, depth, image, rect, visible):
    """The copies in depth order, row by row of each point's tile rect (tx0, ty0, and
    the spans), then stably by tile."""
    offs = np.cumsum([0] + [-(-v.camera.width // tile) * -(-v.camera.height // tile) for v in views])
    grids = np.array([-(-v.camera.width // tile) for v in views])
    tx0, ty0, w, h = (x[depth] for x in rect)
    im, vis = image[depth], visible[depth]
    tiles, pts = [], []
    for dy in range(int(h[vis].max(initial=0)) + 1):
        for dx in range(int(w[vis].max(initial=0)) + 1):
            ok = vis & (w >= dx) & (h >= dy)
            tiles.append(np.where(ok, offs[im] + (ty0 + dy) * grids[im] + tx0 + dx, -1))
            pts.append(depth)
    tiles, pts = np.stack(tiles, 1).ravel(), np.stack(pts, 1).ravel()
    keep = tiles >= 0
    order = np.argsort(tiles[keep], kind="stable")
    keys, vals = r.sorted_copies()
    assert np.array_equal(keys, tiles[keep][order]) and np.array_equal(vals, pts[keep][order])
    # every tile's range of that list (searched for, or scanned on sparsely covered images)
    ranges = r.arr("ranges", np.uint32, 2 * offs[-1]).reshape(-1, 2)
    count = np.bincount(keys, minlength=offs[-1])
    assert np.array_equal(ranges[:, 1] - ranges[:, 0], count)
    assert np.array_equal(ranges[count > 0, 0], np.searchsorted(keys, np.arange(offs[-1])[count > 0]))


# one tile and its edges, one look-back group and its edges (16 tiles of 1024), the change of
# tile size (256 Ki expected elements), several groups of 4096-key tiles
@pytest.mark.parametrize("n", [1, 31, 1023, 1024, 1025, 16384, 16385, 262144, 262145, 1500077])
def test_sorts_at_tile_and_group_edges(n):
    _check([_view(n, 320, 200, "spread", n)])


@pytest.mark.parametrize("depths", ["equal", "two", "culled"])
@pytest.mark.parametrize("n", [5000, 300001])
def test_sorts_with_few_distinct_keys(n, depths):
    _check([_view(n, 160, 96, depths, n)])


def test_sorts_of_several_images_and_wide_tile_ids():
    # 2^18 tiles of 8x8 (9-bit tile digits) beside a small image: image-major depth keys
    _check([_view(70001, 4096, 4096, "spread", 1), _view(3000, 64, 48, "spread", 2)], tile=8)


@pytest.mark.parametrize("tile", [8, 16])
def test_rects_of_several_images_follow_the_depth_sort(tile):
    _check([_view(20011, 320, 200, "spread", 3), _view(7, 64, 48, "spread", 4), _view(300007, 100, 75, "culled", 5)],
           tile=tile)


# small Gaussians (spans of up to two tiles), ones whose spans leave the rect's code (three
# tiles and more), and an image too large for the code (its rects are gathered in depth order)
@pytest.mark.parametrize("width,height,scale,tile", [(320, 200, 0.004, 16), (320, 200, 0.15, 16),
                                                     (4096, 4096, 2e-4, 8)])
@pytest.mark.parametrize("n", [3001, 300001])
def test_gaussian_rects_follow_the_depth_sort(n, width, height, scale, tile):
    if n > 10000 and scale > 0.1:
        n = 20001  # many copies a point
    rng = np.random.default_rng(n + width)
    v = _view(n, width, height, "spread", n)
    v.scale = (v.xyz[:, 2] * scale * rng.uniform(0.2, 1.0, n)).astype(np.float32)
    v.scale[v.scale < 0] = 0.01
    r = Run([v], mode="gaussian", tile=tile, max_copies=400 if scale > 0.1 else 0)
    assert r.status == 0
    rect = r.arr("rect", np.uint32, 2 * n).reshape(n, 2).astype(np.int64)
    tx0, ty0, tx1, ty1 = rect[:, 0] & 0xFFFF, rect[:, 0] >> 16, rect[:, 1] & 0xFFFF, rect[:, 1] >> 16
    visible = tx0 <= tx1
    zb = r.arr("zbits", np.uint32, n).astype(np.int64)
    depth = np.lexsort((np.arange(n), np.where(visible, zb, int(_bits(v.camera.far)))))
    assert np.array_equal(r.arr("depth_sorted", np.uint32, n), depth.astype(np.uint32))
    _check_copies(r, [v], tile, depth, np.zeros(n, np.int64), (tx0, ty0, tx1 - tx0, ty1 - ty0), visible)
