"""Calls in a row on one stream, whose kernels may overlap: each finds what the call
before it wrote."""
import ctypes

import numpy as np
import pytest
import torch

from gpu_util import dev_keys, stream_handle
from paper_2609_00843_gb300 import gen, rtcdf
from test_batched_gpu import check_segments, make_segments

pytestmark = pytest.mark.gpu


# A segmented sort of in-CTA segments only: those over wide ranges keep the first
# launch busy long after the second one has sorted the few others.  The sort after it
# reads what the first launch writes.
@pytest.mark.parametrize("planned", ["host", "device"])
def test_sort_after_a_segmented_sort_without_scan_items(planned):
    s, S, n, R = stream_handle(), 1520, 60_000, 55_000
    lengths = np.full(S, n, np.int64)
    lengths[::100] = 50
    ranges = np.where(lengths == n, R, 100)
    offs = np.concatenate([[0], np.cumsum(lengths)]).astype(np.int64)
    x = dev_keys(int(offs[-1]), 0, 100, gen.UNIFORM, 51)
    for i in range(S):
        if lengths[i] == n:
            gen.keys_device(x.data_ptr() + 4 * int(offs[i]), n, 0, R, gen.UNIFORM, gen.derive_seed(52, i), stream=s)
    out = torch.empty_like(x)
    mn, mx = np.zeros(S, np.int64), ranges
    if planned == "host":
        plan = rtcdf.BatchPlan(offs, mn, mx)
        wsb = plan.workspace_size()
    else:
        meta = [torch.from_numpy(np.ascontiguousarray(v)).cuda() for v in (offs, mn, mx)]
        wsb = rtcdf.rtcdf_batch_device_workspace_size(S, int(offs[-1]), R)
    ws = torch.zeros(wsb // 4, dtype=torch.int32, device="cuda")
    m, at = 24_000, 17_000
    back = torch.empty(m, dtype=torch.int32, device="cuda")
    for i in (1, S // 2 + 1, S - 2) * 6:
        out.fill_(7)
        lo = int(offs[i])
        if planned == "host":
            assert plan.run(x.data_ptr(), out.data_ptr(), ws.data_ptr(), wsb, s) == rtcdf.OK
        else:
            assert rtcdf.rtcdf_sort_batched_device_ws(x.data_ptr(), out.data_ptr(), *[t.data_ptr() for t in meta], S,
                                                      int(offs[-1]), R, ws.data_ptr(), wsb, s) == rtcdf.OK
        assert rtcdf.rtcdf_sort(out.data_ptr() + 4 * (lo + at), back.data_ptr(), m, 0, R, s) == rtcdf.OK
        assert torch.equal(back, x[lo:lo + n].sort().values[at:at + m])
    assert rtcdf.rtcdf_status_get(s) == (rtcdf.OK, 0)
    assert rtcdf.rtcdf_batch_status_get(ws.data_ptr(), s) == (rtcdf.OK, 0)


class Segments:
    """One layout, sorted in the library's workspace of a stream."""

    def __init__(self, lengths, Rs, max_R, stream):
        S = len(lengths)
        self.x, self.offs, self.mn, self.mx = make_segments(lengths, Rs, [-7] * S, [i % 3 for i in range(S)], range(S))
        self.out = torch.empty_like(self.x)
        self.meta = [torch.from_numpy(v).cuda() for v in (self.offs, self.mn, self.mx)]
        self.max_R, self.s = max_R, stream

    def reserve(self):
        assert rtcdf.rtcdf_batch_reserve(len(self.mn), self.x.numel(), self.max_R, self.s) == rtcdf.OK

    def sort(self):
        return rtcdf.rtcdf_sort_batched(self.x.data_ptr(), self.out.data_ptr(), *[t.data_ptr() for t in self.meta],
                                        len(self.mn), self.x.numel(), self.max_R, self.s)

    def check(self, sort):
        self.out.fill_(0x7FFFFFFF)
        torch.cuda.synchronize()
        assert sort() in (None, rtcdf.OK)
        assert rtcdf.rtcdf_status_get(self.s) == (rtcdf.OK, 0)
        check_segments(self.x, self.out, self.offs, self.mn, self.mx)


# The library's workspace is in the layout of the bounds of the sort before, which is a
# call or a graph's replay: the host sees the calls only.  (R: Y is replayed; C: Y is
# captured; the others are calls.)
@pytest.mark.parametrize("order", ["XCYRXRR", "CXRXR", "CYXYRX", "XYCXRZRZYR"])
def test_segmented_sorts_and_replays_with_other_bounds(order):
    stream = torch.cuda.Stream()
    s = stream.cuda_stream
    runs = {"X": Segments([200_001, 70_000, 5, 131_073], [1 << 20, 1 << 16, 3, 70_000], 1 << 20, s),
            "Y": Segments([2000 + 7 * i for i in range(300)] + [70_000], [4096 - i for i in range(300)] + [4096], 4096, s),
            "Z": Segments([66_000, 90_000, 1000], [5000, 4097, 100], 5000, s)}
    for r in runs.values():
        r.reserve()
    graph = torch.cuda.CUDAGraph()

    def replay():
        with torch.cuda.stream(stream):
            graph.replay()

    torch.cuda.synchronize()
    for step in order:
        if step == "C":
            with torch.cuda.graph(graph, stream=stream):
                assert runs["Y"].sort() == rtcdf.OK
        elif step == "R":
            runs["Y"].check(replay)
        else:
            runs[step].check(runs[step].sort)


# A sort whose first launch may overlap the kernel before it in its stream, and whose
# input another stream writes after that kernel: behind an event, and on the legacy
# default stream behind a stream that it waits for by itself.
@pytest.mark.parametrize("n,R", [(20_000, 1000), (1_000_000, 5000), (3_000_001, 50_021), (400_000, 300_000)])
@pytest.mark.parametrize("legacy", [False, True])
def test_sort_of_what_another_stream_writes(n, R, legacy):
    cuda = ctypes.CDLL("libcuda.so.1")
    handle = ctypes.c_void_p()
    assert cuda.cuStreamCreate(ctypes.byref(handle), 0) == 0          # (waits for the legacy stream, and it for this one)
    other = torch.cuda.ExternalStream(handle.value)
    mine = torch.cuda.default_stream() if legacy else torch.cuda.Stream()
    x = [dev_keys(n, 0, R, gen.UNIFORM, gen.derive_seed(53, n, k)) for k in range(2)]
    want = [v.sort().values for v in x]
    a, out = torch.empty_like(x[0]), torch.empty_like(x[0])
    torch.cuda.synchronize()
    for k in (0, 1, 0, 1):
        rtcdf.rtcdf_sort(a.data_ptr(), a.data_ptr(), n, 0, R, mine.cuda_stream)   # the kernel before
        with torch.cuda.stream(other):
            if not legacy:
                other.wait_stream(mine)
            torch.cuda._sleep(400_000)
            a.copy_(x[k])
        if not legacy:
            mine.wait_stream(other)
        assert rtcdf.rtcdf_sort(a.data_ptr(), out.data_ptr(), n, 0, R, mine.cuda_stream) == rtcdf.OK
        torch.cuda.synchronize()
        assert torch.equal(out, want[k])
    rtcdf.rtcdf_status_get(mine.cuda_stream)         # (the first sort's input was never written)
    assert cuda.cuStreamDestroy_v2(handle) == 0
