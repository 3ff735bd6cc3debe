"""The workspace layout names the sorts' look-back words where they lie: over the
backward's partial rows, with room for both."""
import ctypes as ct

import pytest

from paper_2508_19140_gb300 import rast

from test_abi import _fake_view, _opts, lib  # noqa: F401


@pytest.mark.parametrize("mode", [0, 1])
@pytest.mark.parametrize("n,max_copies", [(1, 0), (1025, 0), (300000, 0), (300000, 1), (1000, 4000)])
def test_sort_status_lies_over_the_partial_rows(lib, n, max_copies, mode):  # noqa: F811
    arr = (rast.View * 1)(_fake_view(n=n))
    o = _opts(lib, mode=mode, max_copies=max_copies)
    count = lib.rasterize_workspace_layout(arr, 1, ct.byref(o), None, 0)
    ents = (rast.WsEntry * count)()
    lib.rasterize_workspace_layout(arr, 1, ct.byref(o), ents, count)
    lay = {e.name.decode(): (e.offset, e.bytes) for e in ents}
    assert len(lay) == count
    off, size = lay["sort_status"]
    assert off == lay["partial"][0] and size <= lay["partial"][1]
    tiles = -(-n // (1024 if n <= 1 << 18 else 4096))  # of the depth sort, four passes of 7-bit digits
    assert size >= (0 if tiles == 1 else 4 * 128 * 4 * tiles)
    # every array but the aliases lies apart from the others and inside the workspace
    own = sorted(v for k, v in lay.items() if k not in ("depth_sorted", "sorted_keys", "sorted_vals", "sort_status"))
    for (a, n_a), (b, _) in zip(own, own[1:]):
        assert a % 256 == 0 and a + max(n_a, 1) <= b
    assert own[-1][0] + own[-1][1] <= lib.rasterize_workspace_size(arr, 1, ct.byref(o))
