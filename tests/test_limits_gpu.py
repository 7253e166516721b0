"""Outputs at the limits of the arithmetic: the last positions of the largest
arrays, where 32-bit positions end, counts whose sums pass 2^32, and the longest lists."""
import pytest
import torch

from gpu_util import stream_handle
from paper_2609_00843_gb300 import gen, rtcdf

pytestmark = pytest.mark.gpu

N_MAX = (1 << 32) - 1


def u32(x):
    """The int32 with the bits of the 32-bit unsigned x."""
    return x - (1 << 32) if x >= 1 << 31 else x


def end_window(counts, R, length, offset, ws, wsb):
    """Positions [N_MAX - length, N_MAX) of the array with these counts, written `offset`
    elements into a buffer whose other elements stay -5."""
    s = stream_handle()
    out = torch.full((length + 8,), -5, dtype=torch.int32, device="cuda")
    win = out[offset:offset + length]
    assert rtcdf.rtcdf_fill_from_counts(counts.data_ptr(), N_MAX, 0, R, N_MAX - length, N_MAX, win.data_ptr(),
                                        ws.data_ptr(), wsb, s) == rtcdf.OK
    assert rtcdf.rtcdf_ws_status_get(ws.data_ptr(), s) == (rtcdf.OK, 0)
    assert bool((out[:offset] == -5).all()) and bool((out[offset + length:] == -5).all())
    return win


# Windows that end before their output's first whole vector would begin.
@pytest.mark.parametrize("R", [20_000, 1 << 20])
def test_windows_without_a_whole_vector_at_the_end_of_the_largest_array(R):
    counts = torch.ones(R, dtype=torch.int32, device="cuda")
    counts[0] = u32(N_MAX - (R - 1))
    wsb = rtcdf.rtcdf_workspace_size(R)
    ws = torch.zeros(wsb // 4, dtype=torch.int32, device="cuda")
    for offset in range(4):
        for length in range(1, 8):
            win = end_window(counts, R, length, offset, ws, wsb)
            assert win.tolist() == list(range(R - length, R)), (offset, length)


# A last window of runs that begins within three positions of 2^32: as many runs as
# fill whole windows of the output kernel (of 1024, 2048, 4096, 8192), and one.
@pytest.mark.parametrize("offset", [0, 3])
def test_last_run_of_the_largest_array(offset):
    out = torch.empty(N_MAX + 4, dtype=torch.int32, device="cuda")
    win, s = out[offset:offset + N_MAX], stream_handle()
    for runs in (1024, 2048, 4096, 8192):
        for last in (1, 2):                      # keys of the last run
            R = runs + 1
            counts = torch.ones(R, dtype=torch.int32, device="cuda")
            counts[R - 1] = last
            counts[0] = u32(N_MAX - (R - 2) - last)
            wsb = rtcdf.rtcdf_workspace_size(R)
            ws = torch.zeros(wsb // 4, dtype=torch.int32, device="cuda")
            out.fill_(-5)
            assert rtcdf.rtcdf_fill_from_counts(counts.data_ptr(), N_MAX, 0, R, 0, N_MAX, win.data_ptr(), ws.data_ptr(),
                                                wsb, s) == rtcdf.OK
            assert rtcdf.rtcdf_ws_status_get(ws.data_ptr(), s) == (rtcdf.OK, 0)
            tail = list(range(1, R - 1)) + [R - 1] * last
            assert win[N_MAX - len(tail):].tolist() == tail, (runs, last)
            assert int(torch.count_nonzero(win[:N_MAX - len(tail)])) == 0, (runs, last)
            assert bool((out[:offset] == -5).all()) and bool((out[offset + N_MAX:] == -5).all())


# Runs of one key up to the very last position: scan and output in one launch (R up
# to 16384), and the general kernels' form for short runs.
@pytest.mark.parametrize("R", [301, 16384, 1 << 24])
def test_short_runs_at_the_end_of_the_largest_array(R):
    counts = torch.ones(R, dtype=torch.int32, device="cuda")
    counts[0] = u32(N_MAX - (R - 1))             # value 0 to position 2^32 - R, then a position each
    wsb = rtcdf.rtcdf_workspace_size(R)
    ws = torch.zeros(wsb // 4, dtype=torch.int32, device="cuda")
    for offset in (0, 1, 3):
        for length in (1, 300, 512, 1000, 5003, 70_001):
            win = end_window(counts, R, length, offset, ws, wsb)
            want = torch.arange(R - length, R, device="cuda").clamp_(min=0).int()
            assert torch.equal(win, want), (offset, length)


# Counts that do not add up and whose running sum passes 2^32 on the way, so that the
# run ends decrease: reported, nothing stored outside the window, and the workspace
# serves the next call.  Scan and output in one launch, then the general kernels over
# short runs and over long ones (each with more runs than a window of the kernel).
# The sum falls at value `at` to that of value `to`; one window ends early in the scan's
# chunk of 4096 values with the fall.
@pytest.mark.parametrize("R,each", [(1501, 40), (16384, 40), (20_000, 40), (20_000, 700), (50_000, 3)])
@pytest.mark.parametrize("at,to", [(500, 250), (8192, 1638), (16_484, 1000)])
def test_counts_that_pass_the_largest_sum(R, each, at, to):
    at, to = min(at, R - 500), min(to, R - 600)
    s = stream_handle()
    counts = torch.full((R,), each, dtype=torch.int32, device="cuda")
    counts[at] = u32((1 << 32) - each * (at - to))
    top = each * at                                      # the sum before the fall
    ends = (R - 1 - at + to) * each                      # the last sum
    total = max(top, ends) + 1
    wsb = rtcdf.rtcdf_workspace_size(R)
    ws = torch.zeros(wsb // 4, dtype=torch.int32, device="cuda")
    chunk = at // 4096 * 4096 * each
    windows = [(0, total), (total // 3, total), (total // 2 + 1, total - 5), (top * 3 // 4, top), (total - 3, total)]
    for lo, hi in windows + [(chunk - 1500, chunk + 500)] * (chunk > 0):
        length = hi - lo
        out = torch.full((length + 72,), -5, dtype=torch.int32, device="cuda")
        assert rtcdf.rtcdf_fill_from_counts(counts.data_ptr(), total, 0, R, lo, hi, out[33:].data_ptr(),
                                            ws.data_ptr(), wsb, s) == rtcdf.OK
        assert rtcdf.rtcdf_ws_status_get(ws.data_ptr(), s) == (rtcdf.ERR_KEY_OUT_OF_RANGE, rtcdf.DEV_KEY_OUT_OF_RANGE)
        assert bool((out[:33] == -5).all()) and bool((out[33 + length:] == -5).all())
    counts[at] = each
    out = torch.empty(each * R, dtype=torch.int32, device="cuda")
    assert rtcdf.rtcdf_fill_from_counts(counts.data_ptr(), each * R, 0, R, 0, each * R, out.data_ptr(), ws.data_ptr(),
                                        wsb, s) == rtcdf.OK
    assert rtcdf.rtcdf_ws_status_get(ws.data_ptr(), s) == (rtcdf.OK, 0)
    assert torch.equal(out, torch.arange(R, device="cuda", dtype=torch.int32).repeat_interleave(each))


# The largest segment, its last values in runs of one key: the shares of its last
# output item, the last block of short runs, and (2048 values: a window of the
# kernel) a last run that begins a window at the last position.
@pytest.mark.parametrize("values", [2048, 5000])
@pytest.mark.parametrize("planned", ["host", "device"])
def test_largest_segment(values, planned):
    s, R = stream_handle(), 70_000
    x = torch.zeros(N_MAX, dtype=torch.int32, device="cuda")
    x[torch.arange(1, values + 1, device="cuda") * 800_000] = torch.arange(R - values, R, device="cuda", dtype=torch.int32)
    out = torch.full((N_MAX + 4,), -5, dtype=torch.int32, device="cuda")
    if planned == "host":
        plan = rtcdf.BatchPlan([0, N_MAX], [0], [R])
        wsb = plan.workspace_size()
        ws = torch.zeros(wsb // 4, dtype=torch.int32, device="cuda")
        assert plan.run(x.data_ptr(), out.data_ptr(), ws.data_ptr(), wsb, s) == rtcdf.OK
    else:
        offs, mn, mx = (torch.tensor(v, dtype=torch.int64, device="cuda") for v in ([0, N_MAX], [0], [R]))
        wsb = rtcdf.rtcdf_batch_device_workspace_size(1, N_MAX, R)
        ws = torch.zeros(wsb // 4, dtype=torch.int32, device="cuda")
        assert rtcdf.rtcdf_sort_batched_device_ws(x.data_ptr(), out.data_ptr(), offs.data_ptr(), mn.data_ptr(),
                                                  mx.data_ptr(), 1, N_MAX, R, ws.data_ptr(), wsb, s) == rtcdf.OK
    assert rtcdf.rtcdf_batch_status_get(ws.data_ptr(), s) == (rtcdf.OK, 0)
    assert torch.equal(out[N_MAX - values:N_MAX], torch.arange(R - values, R, device="cuda", dtype=torch.int32))
    assert int(torch.count_nonzero(out[:N_MAX - values])) == 0
    assert bool((out[N_MAX:] == -5).all())


# The partition of so many keys that an item of the bucket kernel lists its slabs twice
# (more than 4096 of 32768 keys; 128 buckets, four items each).
def test_partition_of_more_slabs_than_a_list_holds():
    n, R, mn, s = 600_000_003, 1 << 22, -(1 << 20), stream_handle()
    x = torch.empty(n + 1, dtype=torch.int32, device="cuda")[1:]
    gen.keys_device(x.data_ptr(), n, mn, R, gen.UNIFORM, gen.derive_seed(92, R), stream=s)
    out = torch.empty_like(x)
    assert rtcdf.rtcdf_sort(x.data_ptr(), out.data_ptr(), n, mn, mn + R, s) == rtcdf.OK
    assert rtcdf.rtcdf_status_get(s) == (rtcdf.OK, 0)
    counts = torch.bincount(x.sub_(mn), minlength=R)
    assert torch.equal(out, torch.repeat_interleave(torch.arange(mn, mn + R, device="cuda", dtype=torch.int32), counts))
