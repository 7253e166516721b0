"""Which kernels a sort takes: those of the built-in rules unless the caller, or an
entry of the caller's tuning table for the sort's class, gives parameters."""
import ctypes

import pytest
import torch

from gpu_util import assert_matches_oracle, dev_keys, gpu_sort, stream_handle
from paper_2609_00843_gb300 import gen, rtcdf

pytestmark = pytest.mark.gpu


@pytest.fixture(autouse=True)
def builtin_table():
    yield
    rtcdf.rtcdf_tune_reset()


def launches(n, R, params=None):
    """Kernels of one sort: the nodes of its graph."""
    cuda = ctypes.CDLL("libcuda.so.1")
    x = dev_keys(n, 0, R, gen.UNIFORM, 61)
    out = torch.empty_like(x)
    wsb = rtcdf.rtcdf_workspace_size(R)
    ws = torch.zeros(wsb // 4, dtype=torch.int32, device="cuda")
    s = torch.cuda.Stream()
    gpu_sort(x, 0, R, out)
    torch.cuda.synchronize()
    stream, graph, count = ctypes.c_void_p(s.cuda_stream), ctypes.c_void_p(), ctypes.c_size_t()
    assert cuda.cuStreamBeginCapture_v2(stream, 2) == 0      # (relaxed)
    rc = rtcdf.rtcdf_sort_ex(x.data_ptr(), out.data_ptr(), n, 0, R, params, ws.data_ptr(), wsb, None, s.cuda_stream)
    assert cuda.cuStreamEndCapture(stream, ctypes.byref(graph)) == 0
    assert rc == rtcdf.OK
    assert cuda.cuGraphGetNodes(graph, None, ctypes.byref(count)) == 0
    assert cuda.cuGraphDestroy(graph) == 0
    return count.value


# One CTA; scan and output in one launch; the same over a wide range.
@pytest.mark.parametrize("n,R,own", [(10_007, 1000, 1), (1_000_000, 5000, 2), (1_000_000, 1 << 22, 3)])
def test_a_table_without_an_entry_leaves_the_rules_their_kernels(n, R, own):
    lr, nc = (R - 1).bit_length(), rtcdf.rtcdf_tune_n_class(n)
    entry = rtcdf.Params(fill_threads=512, fill_chunk=8192)
    assert launches(n, R) == own
    for table in ([], [(lr, nc + 1, entry)], [(lr, nc, rtcdf.Params(tile_width=1 << 20))], [(lr, nc, rtcdf.Params())]):
        rtcdf.rtcdf_tune_set(table)
        assert launches(n, R) == own, table
        x = dev_keys(n, -3, R, gen.NORMAL, 62)
        assert_matches_oracle(x, gpu_sort(x, -3, R - 3), -3, R - 3)
    rtcdf.rtcdf_tune_set([(lr, nc, entry)])                  # its own entry: the general kernels
    assert launches(n, R) == launches(n, R, entry) == (4 if R == 1 << 22 else 3)


def test_autotune_times_the_rules_with_their_kernels():
    # The general scan (four chunks) finds a stray ticket in the workspace and reports
    # it; scan and output in one launch have no use for the ticket.
    n, R = 200_000, 1 << 14
    x = dev_keys(n, 0, R, gen.UNIFORM, 63)
    out = torch.empty_like(x)
    wsb = rtcdf.rtcdf_workspace_size(R)
    ws = torch.zeros(wsb // 4, dtype=torch.int32, device="cuda")
    ws[1] = 1                                                # control block word 1: the scan ticket
    cases, s = [(x.data_ptr(), out.data_ptr(), n, 0, R)], stream_handle()
    t, gm, best = rtcdf.rtcdf_autotune(cases, [rtcdf.Params()], 3, ws.data_ptr(), wsb, s)
    assert best == 0 and gm == [1.0] and t[0][0] > 0
    assert_matches_oracle(x, out, 0, R)
    ws.zero_()
    t, gm, best = rtcdf.rtcdf_autotune(cases, [rtcdf.Params(), rtcdf.Params(hist_threads=512)], 3, ws.data_ptr(), wsb, s)
    assert all(v > 0 for v in t[0])


# A histogram alone: several tiles for small arrays over a range that one would hold.
@pytest.mark.parametrize("R", [16_384, 16_385, 32_768, 32_769, 57_344, 57_345])
@pytest.mark.parametrize("n", [1, 70_003, (1 << 20) - 1, 1 << 20])
def test_histogram_alone(R, n):
    x = torch.empty(n + 1, dtype=torch.int32, device="cuda")[1:]
    gen.keys_device(x.data_ptr(), n, -4, R, gen.NORMAL, gen.derive_seed(64, R, n), stream=stream_handle())
    counts = torch.zeros(R, dtype=torch.int32, device="cuda")
    for k in (1, 2):
        assert rtcdf.rtcdf_hist_accumulate(x.data_ptr(), n, -4, R - 4, counts.data_ptr(), stream_handle()) == rtcdf.OK
        assert torch.equal(counts.long(), k * torch.bincount(x + 4, minlength=R))
