"""The Gaussian gradient reduction's two ways through the points: each thread its
own point, where the backward replayed more than about a copy a point, and only
the points with a replayed copy collected for full warps, where it replayed
fewer. All four gradients against the FP64 oracle (bars of test_gpu_parity.py,
without the points that touch a pixel whose termination is within 1e-5 of the
threshold), and the points with a gradient are exactly the oracle's."""
import numpy as np
import pytest
import torch

import oracle

from gpu_util import Run
from test_gpu_gauss_lists import _view
from test_gpu_parity import _check_grad

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _need_gpu():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2508_19140_gb300 import build
    build.build()
    oracle.build()


def _keep(v, kw):
    """Points none of whose pixels is near the termination threshold."""
    near = oracle.render(v.xyz, v.opacity, v.feat, v.camera, scale=v.scale, **kw)["margin"] <= 1e-5
    p = oracle.project(v.xyz, v.camera, scale=v.scale, **kw)
    keep = np.ones(len(v.xyz), bool)
    for i in np.nonzero(p["vis"])[0]:
        x0, x1, y0, y1 = p["box"][i]
        keep[i] = not near[y0:y1 + 1, x0:x1 + 1].any()
    return keep


def _check(v, tile, collected, dilation=0.16, skip=()):
    n, c = v.feat.shape
    r = Run([v], mode="gaussian", tile=tile, backward=True, max_copies=64, dilation=dilation)
    assert r.status == 0
    kw = dict(mode="gaussian", gauss_cov="ewa", tile=tile, pin32=True, dilation=dilation)
    replayed = int(r.stats["needed_records"])  # the backward replays what the forward read
    assert (8 * replayed <= n * (9 if c <= 4 else 12)) == collected
    keep = _keep(v, kw)
    keep[list(skip)] = False
    assert keep.sum() > 0.5 * n
    ref = oracle.backward(v.xyz, v.opacity, v.feat, v.camera, v.g_feat, v.g_alpha, v.g_depth, scale=v.scale, **kw)
    g = r.grads()
    has = np.abs(ref["d_feat"]).sum(1) > 0
    assert np.array_equal((np.abs(g["d_feat"]).sum(1) > 0)[keep], has[keep])
    assert has[keep].any() and not has.all()
    _check_grad(g["d_feat"], ref["d_feat"], mask=keep)
    for k in ("d_opacity", "d_xyz", "d_scale"):
        _check_grad(g[k], ref[k], norm=1e-4, er=1e-3, ea=1e-5, mask=keep)
        assert np.all(g[k][keep & ~has] == 0), k
    return r


# dense clouds: most points lie behind the early termination
@pytest.mark.parametrize("tile", [8, 16])
@pytest.mark.parametrize("c", [1, 4, 16])
@pytest.mark.parametrize("n", [40000, 40033])
def test_collected_points(n, c, tile):
    _check(_view(n, 48, 40, 9, (0.6, 0.95), c), tile, True)


# the same with splats of many tiles, beyond the four whose cutoffs are read first
@pytest.mark.parametrize("c", [4, 16])
def test_collected_points_with_many_copies(c):
    v = _view(6000, 48, 40, 3, (0.9, 0.99), c)
    v.scale[::7] *= 8.0
    _check(v, 8, True)


# thin clouds, and clouds of large splats: more than a replayed copy a point
@pytest.mark.parametrize("tile", [8, 16])
@pytest.mark.parametrize("c", [1, 4, 16])
@pytest.mark.parametrize("n", [255, 257, 3001])
def test_every_point_taken(n, c, tile):
    v = _view(n, 160, 128, 5, (0.02, 0.1), c)
    v.scale[:] = 0.1
    v.xyz[0] = [0.0, 0.0, -1.0]  # behind the camera
    _check(v, tile, False)


def test_two_points_a_thread():
    # 16 channels and 512 Ki points: the gradients of the first points equal those of a smaller cloud
    # that ends with the same points far behind (every later point lies behind the termination)
    n = 512 * 1024 + 77
    v = _view(n, 24, 16, 2, (0.9, 0.99), 16)
    order = np.argsort(v.xyz[:, 2], kind="stable")
    for k in ("xyz", "opacity", "feat", "scale"):
        setattr(v, k, np.ascontiguousarray(getattr(v, k)[order]))
    a = Run([v], mode="gaussian", backward=True)
    m = 100000
    w = _view(m, 24, 16, 2, (0.9, 0.99), 16)
    for k in ("xyz", "opacity", "feat", "scale"):
        setattr(w, k, getattr(v, k)[:m])
    w.g_feat, w.g_alpha, w.g_depth = v.g_feat, v.g_alpha, v.g_depth
    b = Run([w], mode="gaussian", backward=True)
    assert a.status == 0 and b.status == 0
    for x, y in zip(a.image(), b.image()):
        assert np.array_equal(x, y)  # nothing behind the first m points is seen
    assert 12 * n >= 8 * int(a.stats["needed_records"])
    for k, g in a.grads().items():
        assert np.array_equal(g[:m], b.grads()[k]), k
        assert np.all(g[m:] == 0), k


def test_singular_covariance_without_dilation():
    # without dilation a point of scale 0 on a pixel centre has a singular covariance: it covers one
    # pixel, blends nothing, and the chain rule's 0 / 0 gives NaN whether its tile was replayed up to it or not
    for n, collected in ((40000, True), (300, False)):
        v = _view(n, 48, 40, 9, (0.6, 0.95) if collected else (0.02, 0.1), 4)
        if not collected:
            v.scale[:] = 0.2
        for i, z in ((0, 1.0), (1, 8.0)):
            v.xyz[i] = [-z / 8, -z / 8, z]  # screen position (16.5, 12.5), exactly
            v.scale[i] = 0.0
        r = _check(v, 16, collected, dilation=0.0, skip=(0, 1))
        g = r.grads()
        assert np.all(g["d_feat"][:2] == 0) and np.all(g["d_opacity"][:2] == 0)
        assert np.all(np.isnan(g["d_xyz"][:2])) and np.all(np.isnan(g["d_scale"][:2]))


@pytest.mark.parametrize("tile", [8, 16])
@pytest.mark.parametrize("n", [1, 31, 63, 64, 65, 127, 128, 129, 192, 193, 384, 385, 513])
def test_gradients_of_short_lists(n, tile):
    """Lists at the edges of the blends' batches, with a gradient comparison that no near pixel skips."""
    v = _view(n, 8, 8, n)
    kw = dict(mode="gaussian", gauss_cov="ewa", tile=tile, pin32=True)
    keep = _keep(v, kw)
    assert 2 * keep.sum() >= n
    r = Run([v], mode="gaussian", tile=tile, backward=True)
    assert r.status == 0
    ref = oracle.backward(v.xyz, v.opacity, v.feat, v.camera, v.g_feat, v.g_alpha, v.g_depth, scale=v.scale, **kw)
    g = r.grads()
    _check_grad(g["d_feat"], ref["d_feat"], mask=keep)
    for k in ("d_opacity", "d_xyz", "d_scale"):
        _check_grad(g[k], ref[k], norm=1e-4, er=1e-3, ea=1e-5, mask=keep)
