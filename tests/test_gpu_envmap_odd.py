"""The background map's gradient where its sums cannot be converted as 16-byte
vectors: maps of an odd number of values, and a gradient or scratch that is not
16-byte aligned. Against the FP64 oracle with the bars of test_gpu_envmap.py, and
bit for bit against the vector conversion where both can run."""
import numpy as np
import pytest
import torch

import oracle
from paper_2508_19140_gb300 import rast, scenes

from test_gpu_envmap import DEV, _cam, _inputs, _t

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _need_gpu():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2508_19140_gb300 import build
    build.build()
    oracle.build()


def _map_grad(cam, env_np, alpha, g, shift=0, scratch_shift=0):
    """dL/dmap written `shift` floats, from sums kept `scratch_shift` bytes, past an aligned address."""
    env = _t(env_np)
    e = rast.make_envmap(env)
    size = rast.rasterize_bg_scratch_size(e)
    scratch = torch.empty(size + scratch_shift, dtype=torch.uint8, device=DEV)[scratch_shift:]
    buf = torch.full((env.numel() + shift + 1,), 7.0, device=DEV)
    dm = buf[shift: shift + env.numel()].view(env.shape)
    ga = torch.zeros(alpha.shape, device=DEV)
    rast.rasterize_bg_composite_bwd(rast.make_camera(cam), e, None, _t(alpha), _t(g), ga, dm, scratch)
    torch.cuda.synchronize()
    assert torch.all(buf[:shift] == 7.0) and buf[-1] == 7.0  # nothing beside the map
    return dm.cpu().numpy()


# poles, the seam (yaw 180), and a plain view; odd, even and small maps
@pytest.mark.parametrize("yaw,pitch", [(20.0, 5.0), (180.0, 0.0), (90.0, -85.0), (-120.0, 85.0)])
@pytest.mark.parametrize("c,h,w", [(3, 33, 51), (3, 32, 64), (1, 17, 35), (2, 9, 17), (1, 2, 3)])
def test_map_gradient_of_odd_maps(yaw, pitch, c, h, w):
    cam = _cam(97, 61, yaw, pitch)
    env = scenes.env_map(height=h, width=w, c=c)
    _, alpha, g = _inputs(61, 97, c, seed=c + h)
    dm = _map_grad(cam, env, alpha, g)
    _, ref = oracle.env_backward(env, cam, alpha, g)
    assert np.linalg.norm(dm - ref) / np.linalg.norm(ref) < 1e-3
    assert np.all(np.abs(dm[ref == 0]) <= 1e-3 * np.abs(ref).max())  # a coordinate may round across a texel


@pytest.mark.parametrize("c", [1, 4])
@pytest.mark.parametrize("shift,scratch_shift", [(1, 0), (2, 0), (3, 0), (0, 8), (1, 8)])
def test_unaligned_gradient_or_scratch(c, shift, scratch_shift):
    cam = _cam(97, 61, 20.0, 5.0)
    env = scenes.env_map(height=32, width=64, c=c)
    _, alpha, g = _inputs(61, 97, c, seed=c)
    a = _map_grad(cam, env, alpha, g)
    b = _map_grad(cam, env, alpha, g, shift, scratch_shift)
    assert np.array_equal(a.view(np.uint32), b.view(np.uint32))
