"""The Gaussian forward's staging ring on 8x8 tiles, whose batches hold 64 records:
list lengths at the edges of a batch and of the ring of three, and lists whose
pixels all terminate inside a batch, so that warps leave the rest of it. Bars as
in test_gpu_gauss_lists.py."""
import numpy as np
import pytest
import torch

import oracle

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
