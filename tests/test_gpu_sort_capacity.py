"""The tile sort where copies are many more or fewer than its launch shape expects:
few points with a large capacity (4096-key tiles), and few points with many
copies in a capacity of up to 2 Mi (1024-key tiles). Exact, as in
test_gpu_sort.py."""
import numpy as np
import pytest
import torch

from gpu_util import Run
from test_gpu_sort import _bits, _check_copies, _view

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _need_gpu():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2508_19140_gb300 import build
    build.build()


# (points, copies a point may make, splat size): capacities of 2 Mi, one point more, and far above;
# copies from fewer than points to nearly all of the capacity
@pytest.mark.parametrize("n,max_copies,scale", [(131072, 16, 0.002), (131072, 16, 0.012), (131073, 16, 0.012),
                                                (3001, 4000, 0.002), (3001, 4000, 0.15), (17, 2000000, 0.3),
                                                (1500, 1398, 0.5)])
def test_copies_beside_the_expected_count(n, max_copies, scale):
    rng = np.random.default_rng(n)
    v = _view(n, 320, 200, "spread", n)
    v.scale = (v.xyz[:, 2] * scale * rng.uniform(0.2, 1.0, n)).astype(np.float32)
    r = Run([v], mode="gaussian", tile=8, max_copies=max_copies)
    assert r.status == 0
    rect = r.arr("rect", np.uint32, 2 * n).reshape(n, 2).astype(np.int64)
    tx0, ty0, tx1, ty1 = rect[:, 0] & 0xFFFF, rect[:, 0] >> 16, rect[:, 1] & 0xFFFF, rect[:, 1] >> 16
    visible = tx0 <= tx1
    depth = np.lexsort((np.arange(n), np.where(visible, r.arr("zbits", np.uint32, n).astype(np.int64),
                                               int(_bits(v.camera.far)))))
    _check_copies(r, [v], 8, depth, np.zeros(n, np.int64), (tx0, ty0, tx1 - tx0, ty1 - ty0), visible)
