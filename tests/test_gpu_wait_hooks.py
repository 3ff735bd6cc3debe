"""Failure detection without a fault, for the waits of the forward pass on copies
into shared memory: the test hooks withhold one copy, the bounded wait on it runs
out, the call returns and reports RAST_ERR_TIMEOUT, and an ordinary call on the
same workspace right after gives the same bits as one before."""
import numpy as np
import pytest
import torch

from paper_2508_19140_gb300 import rast, scenes

from gpu_util import Run
from test_gpu_gauss_lists import _view

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _need_gpu():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2508_19140_gb300 import build
    build.build()


def _same_again(r, before):
    """An ordinary call on the workspace of the failed one."""
    r.opts.flags = 0
    rast.rasterize_batch(r.cviews, rast.PASS_FWD | rast.PASS_BWD, r.opts, r.ws)
    assert rast.rasterize_get_status(r.ws)[0] == 0
    for a, b in zip(r.image(), before.image()):
        assert np.array_equal(a, b)
    for k, g in before.grads().items():
        assert np.array_equal(r.grads()[k], g), k


@pytest.mark.parametrize("tile", [8, 16])
@pytest.mark.parametrize("opacity", [(0.001, 0.01), (0.3, 0.95)])  # long walks, and tiles that finish early
def test_gauss_forward_wait_runs_out(tile, opacity):
    v = _view(6000, 40, 24, 5, opacity)
    before = Run([v], mode="gaussian", tile=tile, backward=True)
    assert before.status == 0
    r = Run([v], mode="gaussian", tile=tile, backward=True, flags=rast.FLAG_TEST_FWD_BLEND_STALL, ws_fill=0xFF)
    assert r.status == rast.RAST_ERR_TIMEOUT
    assert r.stats["n_copies"] == before.stats["n_copies"]  # everything before the blend is untouched
    _same_again(r, before)


# one tile of the sort (its own wait alone can raise the error), several of 1024 keys, several of 4096;
# bilinear and Gaussian points (their rects travel with the sort in both)
@pytest.mark.parametrize("flag", [rast.FLAG_TEST_KEY_COPY_STALL, rast.FLAG_TEST_VALUE_COPY_STALL])
@pytest.mark.parametrize("mode", ["bilinear", "gaussian"])
@pytest.mark.parametrize("n", [500, 20000, 300000])
def test_sort_copy_wait_runs_out(n, mode, flag):
    v = _view(n, 96, 64, 31) if mode == "gaussian" else scenes.random_small_view(31, n, 96, 64)
    before = Run([v], mode=mode, backward=True)
    assert before.status == 0
    r = Run([v], mode=mode, backward=True, flags=flag, ws_fill=0xFF)
    assert r.status == rast.RAST_ERR_TIMEOUT
    assert r.stats["n_copies"] == 0
    for x in r.image():
        assert np.all(x == 0)
    for k, g in r.grads().items():
        assert np.all(g == 0), k
    _same_again(r, before)


def test_look_back_wait_runs_out_with_two_tiles():
    # 1025 points: two tiles of 1024 keys
    v = scenes.random_small_view(31, 1025, 96, 64)
    r = Run([v], backward=True, flags=rast.FLAG_TEST_SORT_STALL, ws_fill=0xFF)
    assert r.status == rast.RAST_ERR_TIMEOUT and r.stats["n_copies"] == 0
    _same_again(r, Run([v], backward=True))
