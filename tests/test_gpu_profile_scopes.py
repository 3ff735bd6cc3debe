"""The profiler names a stage by the kernel that ran: frames whose tile rects do
not travel with the depth sort gather them, and large, sparsely covered images
scan for their tile ranges."""
import pytest
import torch

from paper_2508_19140_gb300 import rast

from gpu_util import Run
from test_gpu_sort import _view

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _need_gpu():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2508_19140_gb300 import build
    build.build()


@pytest.mark.parametrize("mode", ["bilinear", "gaussian"])
@pytest.mark.parametrize("width,height,gathered,scanned", [(96, 64, False, False), (4096, 4096, True, True)])
def test_stage_names_say_which_kernel_ran(mode, width, height, gathered, scanned):
    v = _view(3001, width, height, "spread", 3)
    v.scale = v.xyz[:, 2] * 2e-4
    rast.rasterize_profile_enable(True)
    r = Run([v], mode=mode, tile=8)
    names = set(rast.rasterize_profile_read())
    rast.rasterize_profile_enable(False)
    assert r.status == 0
    assert ("dup.gather" in names, "dup.count" in names) == (gathered, not gathered)
    assert ("ranges.scan" in names, "ranges" in names) == (scanned, not scanned)
