"""What an autograd node keeps from the forward for the backward: cameras and
options of the call, and no view with its device pointers."""
import numpy as np
import pytest
import torch

from paper_2508_19140_gb300 import rast, scenes

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


@pytest.fixture(scope="module", autouse=True)
def _need_gpu():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2508_19140_gb300 import build
    build.build()


def _run(v, between=None):
    xyz = torch.from_numpy(v.xyz).to(DEV)
    op, feat = (torch.from_numpy(a).to(DEV).requires_grad_(True) for a in (v.opacity, v.feat))
    images = rast.rasterize(xyz, op, feat, v.camera)
    if between:
        between(images)
    grads = torch.autograd.grad(images, [feat, op], [torch.from_numpy(g).to(DEV)
                                                     for g in (v.g_feat, v.g_alpha, v.g_depth)])
    return [g.cpu().numpy() for g in grads]


def test_no_view_is_kept():
    v = scenes.random_small_view(5, 2000, 96, 64)

    def look(images):
        for cam in images[0].grad_fn.c_cams:
            assert isinstance(cam, rast.Camera) and cam._b_base_ is None  # its own memory, no view behind it

    _run(v, look)


def test_the_backward_sees_the_camera_of_its_forward():
    v = scenes.random_small_view(5, 2000, 96, 64)
    before = _run(v)
    fx, t = v.camera.fx, np.array(v.camera.t, copy=True)

    def move(_):
        v.camera.fx = 2.0 * fx
        v.camera.t = t + 1.0

    moved = _run(v, move)
    v.camera.fx, v.camera.t = fx, t
    for a, b in zip(before, moved):
        assert np.array_equal(a, b)
