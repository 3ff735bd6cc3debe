"""The Gaussian forward's staging ring: list lengths at the edges of its batches (128
records, or 64 on 8x8 tiles of large images) and of the ring of three, and
lists whose pixels all terminate inside a batch, so that warps leave the rest of
it. Bars as in test_gpu_gauss_lists.py."""
import numpy as np
import pytest
import torch

import oracle
from paper_2508_19140_gb300 import scenes

from gpu_util import Run
from test_gpu_gauss_lists import _check, _view

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _need_gpu():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2508_19140_gb300 import build
    build.build()
    oracle.build()


@pytest.mark.parametrize("n", [32, 33, 63, 64, 65, 191, 192, 193, 256, 257])
def test_list_lengths_at_batch_edges(n):
    _check(_view(n, 8, 8, n), 8, backward=True)


# every splat covers the whole image, so a pixel terminates after about (0.9: 5, 0.5: 14, 0.1: 88) records
@pytest.mark.parametrize("tile", [8, 16])
@pytest.mark.parametrize("opacity", [0.9, 0.5, 0.1])
@pytest.mark.parametrize("n", [40, 140, 700])
def test_termination_inside_a_batch(n, opacity, tile):
    v = _view(n, 21, 19, n, (opacity, opacity + 0.05))
    v.scale[:] = 5.0
    _check(v, tile)


@pytest.mark.parametrize("c", [1, 16])
def test_widest_and_narrowest_records(c):
    _check(_view(900, 40, 24, 7, c=c), 8)


def test_both_tile_sizes_blend_the_same_pixels():
    v = _view(3000, 61, 43, 11, (0.3, 0.95))
    a, b = (Run([v], mode="gaussian", tile=t) for t in (8, 16))
    for x, y in zip(a.image(), b.image()):
        assert np.array_equal(x, y)


LENGTHS = [1, 31, 32, 33, 63, 64, 65, 127, 128, 129, 191, 192, 193, 255, 256, 257, 321, 700]


@pytest.mark.parametrize("c", [1, 4, 16])
@pytest.mark.parametrize("opacity", [(0.01, 0.05), (0.3, 0.6)])
def test_short_batches_of_a_large_image(c, opacity):
    """16900 tiles of 8x8, most of them empty; one tile for each list length, its splats inside it."""
    size, f = 1040, 900.0
    rng = np.random.default_rng(c)
    n = sum(LENGTHS)
    tile = np.repeat(np.arange(len(LENGTHS)), LENGTHS)
    u = 64.0 + 48 * tile + rng.uniform(3.0, 5.0, n)   # 8x8 tile (8 + 6 t, 5 + 7 t)
    w = 40.0 + 56 * tile + rng.uniform(3.0, 5.0, n)
    z = rng.uniform(1.5, 4.0, n)
    xyz = np.stack([(u - size / 2) / f * z, (w - size / 2) / f * z, z], 1).astype(np.float32)
    g = [rng.standard_normal(s).astype(np.float32) for s in ((size, size, c), (size, size), (size, size))]
    v = scenes.View(xyz=xyz, opacity=rng.uniform(*opacity, n).astype(np.float32),
                    feat=rng.random((n, c)).astype(np.float32), camera=scenes.identity_camera(size, size, f),
                    scale=(z * rng.uniform(0.2, 0.6, n) / f).astype(np.float32), g_feat=g[0], g_alpha=g[1],
                    g_depth=g[2])
    r = _check(v, 8, backward=True)
    counts = np.bincount(r.sorted_copies()[0], minlength=130 * 130)
    assert np.array_equal(counts[[(5 + 7 * t) * 130 + 8 + 6 * t for t in range(len(LENGTHS))]], LENGTHS)
    for x, y in zip(r.image(), Run([v], mode="gaussian", tile=16).image()):
        assert np.array_equal(x, y)
