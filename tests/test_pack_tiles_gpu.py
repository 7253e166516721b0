"""Inputs that the packed histogram leaves to the range tiles, in turn with inputs that
it counts itself: in one workspace, in place, and in a graph."""
import pytest
import torch

from gpu_util import dev_keys, stream_handle
from paper_2609_00843_gb300 import gen, rtcdf

pytestmark = pytest.mark.gpu


# By range tiles of a launch of their own, from its fewest keys on (one tile, five,
# seven), and in the packed histogram's launch.
@pytest.mark.parametrize("R,n", [(57_344, 1_000_000_001), (1 << 18, 200_000_000), (360_448, 143_000_001),
                                 (65_536, 500_000_003), (1 << 18, 199_999_999), (1 << 18, 20_000_000)])
@pytest.mark.parametrize("in_place", [False, True])
def test_packed_and_tiled_inputs_in_turn(R, n, in_place):
    s = torch.cuda.Stream()
    inputs = [dev_keys(n, -9, R, gen.UNIFORM, 71), dev_keys(n, -9, R, gen.UNIFORM, 72).sort().values]
    inputs.append(torch.where(torch.arange(n, device="cuda") % 5 < 2, R - 10, -9 + R // 3).int())   # two keys
    counts = [torch.bincount(x + 9, minlength=R) for x in inputs]
    want = [torch.repeat_interleave(torch.arange(-9, R - 9, device="cuda", dtype=torch.int32), c) for c in counts]
    x = torch.empty(n, dtype=torch.int32, device="cuda")
    out = x if in_place else torch.empty_like(x)
    wsb = rtcdf.rtcdf_workspace_size(R)
    ws = torch.zeros(wsb // 4, dtype=torch.int32, device="cuda")

    def sort():
        return rtcdf.rtcdf_sort_ws(x.data_ptr(), out.data_ptr(), n, -9, R - 9, ws.data_ptr(), wsb, s.cuda_stream)

    graph = torch.cuda.CUDAGraph()
    for k in (0, 1, 0, 2, 1):
        x.copy_(inputs[k])
        torch.cuda.synchronize()
        assert sort() == rtcdf.OK
        torch.cuda.synchronize()
        assert torch.equal(out, want[k])
    with torch.cuda.graph(graph, stream=s):
        assert sort() == rtcdf.OK
    for k in (2, 0, 1, 0):
        x.copy_(inputs[k])
        torch.cuda.synchronize()
        with torch.cuda.stream(s):
            graph.replay()
        torch.cuda.synchronize()
        assert torch.equal(out, want[k])
    assert rtcdf.rtcdf_ws_status_get(ws.data_ptr(), s.cuda_stream) == (rtcdf.OK, 0)
