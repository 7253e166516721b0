"""Sorts from several host threads at once, a stream each."""
import threading

import pytest
import torch

from paper_2609_00843_gb300 import gen, rtcdf

pytestmark = pytest.mark.gpu


# The shared memory of a launch depends on n and R, and so must not depend on what
# another thread launches meanwhile: packed counters, partitions with few and with
# many buckets, long inputs over one tile.
@pytest.mark.parametrize("n,ranges,calls", [
    (18_000_000, (180_000, 350_000), 200), (3_000_000, (1 << 22, 1 << 24), 400), (4_100_000, (3 << 20, 4 << 20), 400),
    (200_000_001, (300, 49_152), 60),
])
def test_threads_with_other_ranges(n, ranges, calls):
    x, want, out = [], [], []
    for k, R in enumerate(ranges):
        x.append(torch.empty(n, dtype=torch.int32, device="cuda"))
        gen.keys_device(x[k].data_ptr(), n, -5, R, gen.UNIFORM, gen.derive_seed(91, R),
                        stream=torch.cuda.current_stream().cuda_stream)
        want.append(x[k].sort().values)
        out.append(torch.empty_like(x[k]))
    torch.cuda.synchronize()
    start, codes = threading.Barrier(len(ranges)), [set() for _ in ranges]

    def work(k):
        torch.cuda.set_device(0)
        s = torch.cuda.Stream()
        start.wait()
        for _ in range(calls):
            codes[k].add(rtcdf.rtcdf_sort(x[k].data_ptr(), out[k].data_ptr(), n, -5, ranges[k] - 5, s.cuda_stream))
        s.synchronize()
        codes[k].add(rtcdf.rtcdf_status_get(s.cuda_stream)[0])

    threads = [threading.Thread(target=work, args=(k,)) for k in range(len(ranges))]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert codes == [{rtcdf.OK}] * len(ranges)
    for k in range(len(ranges)):
        assert torch.equal(out[k], want[k])
