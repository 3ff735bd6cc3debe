"""Gaussian blends at the list lengths where their staging changes: empty and
short lists, the edges of a 128-record batch and of the ring of three, lists of
many batches whose warps finish at different times, and points without any
replayed copy in the gradient reduction (with non-finite scales beside them).
Bars as in test_gpu_parity.py: 1e-5 relative + 1e-7 absolute on the images
outside pixels whose termination is within 1e-5 of the threshold, gradients
normwise 1e-4 (features 1e-5)."""
import numpy as np
import pytest
import torch

import oracle
from paper_2508_19140_gb300 import scenes

from gpu_util import Run
from test_gpu_parity import ATOL, RTOL, _check_grad

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _need_gpu():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2508_19140_gb300 import build
    build.build()
    oracle.build()


def _view(n, width, height, seed, opacity=(0.02, 0.3), c=4):
    rng = np.random.default_rng(seed)
    f = 60.0
    z = rng.uniform(1.5, 4.0, n)
    u, w = rng.uniform(1.0, width - 1.0, n), rng.uniform(1.0, height - 1.0, n)
    xyz = np.stack([(u - width / 2) / f * z, (w - height / 2) / f * z, z], 1).astype(np.float32)
    g = [rng.standard_normal(s).astype(np.float32) for s in ((height, width, c), (height, width), (height, width))]
    return scenes.View(xyz=xyz, opacity=rng.uniform(*opacity, n).astype(np.float32),
                       feat=rng.random((n, c)).astype(np.float32), camera=scenes.identity_camera(width, height, f),
                       scale=np.exp(rng.uniform(np.log(5e-3), np.log(5e-2), n)).astype(np.float32),
                       g_feat=g[0], g_alpha=g[1], g_depth=g[2])


def _check(v, tile, backward=False):
    r = Run([v], mode="gaussian", tile=tile, backward=backward)
    assert r.status == 0
    kw = dict(mode="gaussian", gauss_cov="ewa", tile=tile, pin32=True)
    ref = oracle.render(v.xyz, v.opacity, v.feat, v.camera, scale=v.scale, **kw)
    ok = ref["margin"] > 1e-5
    F, A, D = r.image()
    np.testing.assert_allclose(F[ok], ref["F"][ok], rtol=RTOL, atol=ATOL)
    np.testing.assert_allclose(A[ok], ref["alpha"][ok], rtol=RTOL, atol=ATOL)
    np.testing.assert_allclose(D[ok], ref["depth"][ok], rtol=RTOL, atol=10 * ATOL)
    _, last = r.pixel_state()
    assert np.array_equal(last[ok], ref["last_pos"][ok].astype(np.uint32))
    if ok.all():
        assert int(r.stats["needed_records"]) == ref["needed"]
        if backward:
            g = oracle.backward(v.xyz, v.opacity, v.feat, v.camera, v.g_feat, v.g_alpha, v.g_depth, scale=v.scale,
                                **kw)
            got = r.grads()
            _check_grad(got["d_feat"], g["d_feat"])
            for k in ("d_opacity", "d_xyz", "d_scale"):
                _check_grad(got[k], g[k], norm=1e-4, er=1e-3, ea=1e-5)
    return r


@pytest.mark.parametrize("tile", [8, 16])
@pytest.mark.parametrize("n", [1, 31, 127, 128, 129, 384, 385, 513])
def test_list_lengths_at_batch_edges(n, tile):
    _check(_view(n, 8, 8, n), tile, backward=True)  # one tile: its list holds every point


@pytest.mark.parametrize("tile", [8, 16])
@pytest.mark.parametrize("opacity", [(0.001, 0.01), (0.3, 0.95)])
def test_deep_lists_with_and_without_termination(opacity, tile):
    _check(_view(6000, 40, 24, 5, opacity, c=3), tile)


# a thin cloud (every point replayed) and a dense one (most points behind the termination)
@pytest.mark.parametrize("n,width,height", [(5000, 96, 64), (40000, 48, 40)])
def test_points_without_replayed_copies(n, width, height):
    v = _view(n, width, height, 9, (0.6, 0.95))
    a = Run([v], mode="gaussian", backward=True, max_copies=30)
    assert a.status == 0
    unseen = np.abs(a.grads()["d_feat"]).sum(1) == 0
    assert unseen.sum() > n // 2 or n == 5000
    for k in ("d_opacity", "d_xyz", "d_scale"):
        assert np.all(a.grads()[k][unseen] == 0), k
    # two scales that are not finite, behind everything: the chain rule's NaN there, nothing elsewhere
    w = _view(n, width, height, 9, (0.6, 0.95))
    far = np.argsort(-w.xyz[:, 2])[:2]
    w.scale[far] = [np.nan, np.inf]
    b = Run([w], mode="gaussian", backward=True, max_copies=30)
    assert b.status == 0
    keep = np.ones(n, bool)
    keep[far] = False
    for k, g in b.grads().items():
        assert np.all(np.isfinite(g[keep])), k
    assert np.all(np.isnan(b.grads()["d_scale"][far]))
