"""Sorts of ranges wider than one shared-memory tile, at the sizes where the
histogram's kernels change form: against the CPU oracle, element by element."""
import numpy as np
import pytest
import torch

from gpu_util import assert_matches_oracle, dev_keys, gpu_sort, stream_handle
from paper_2609_00843_gb300 import gen, rtcdf

pytestmark = pytest.mark.gpu


# Buckets of 2^15 values: one more than the widest of each counter layout (64,
# 128 buckets), a last bucket of one value, the widest range; lengths with and
# without keys before and after the whole vectors, and a last slab of few keys.
@pytest.mark.parametrize("R,n,offset", [
    (1 << 19, 8_000_001, 1), ((1 << 20) + 1, 3_100_000, 0), (64 << 15, 2_000_003, 3), ((64 << 15) + 1, 1_400_006, 2),
    (128 << 15, 1_000_000, 0), ((128 << 15) + 5, 900_001, 1), ((1 << 24) - 1, 500_000, 2), (1 << 24, 16384 * 700 + 9, 0),
])
@pytest.mark.parametrize("dist", [gen.UNIFORM, gen.NORMAL, gen.ALL_EQUAL])
def test_partitioned_histogram(R, n, offset, dist):
    mn = -(1 << 31) if dist == gen.UNIFORM else 5 - R
    x = torch.empty(n + offset, dtype=torch.int32, device="cuda")[offset:]
    gen.keys_device(x.data_ptr(), n, mn, R, dist, gen.derive_seed(31, R, n), stream=stream_handle())
    out = torch.full((n + 3,), 77, dtype=torch.int32, device="cuda")[3 - offset:3 - offset + n]
    gpu_sort(x, mn, mn + R, out)
    assert_matches_oracle(x, out, mn, mn + R)


def test_partitioned_histogram_of_sorted_and_two_valued_keys():
    n, R = 6_000_000, 1 << 20
    x = dev_keys(n, 0, R, gen.UNIFORM, 5).sort().values
    assert_matches_oracle(x, gpu_sort(x, 0, R), 0, R)
    x = torch.where(torch.arange(n, device="cuda") % 3 == 0, R - 1, 0).int()
    assert_matches_oracle(x, gpu_sort(x, 0, R), 0, R)


def test_partitioned_histogram_in_place_and_in_a_graph():
    n, R, mn = 5_000_000, 1 << 20, -9
    x = dev_keys(n, mn, R, gen.NORMAL, 6)
    want = gpu_sort(x, mn, mn + R)
    assert_matches_oracle(x, want, mn, mn + R)
    y = x.clone()
    gpu_sort(y, mn, mn + R, y)  # no scratch: the range-tile histogram
    assert torch.equal(y, want)
    s = torch.cuda.Stream()
    assert rtcdf.rtcdf_reserve(R, s.cuda_stream) == rtcdf.OK
    torch.cuda.synchronize()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g, stream=s):
        assert rtcdf.rtcdf_sort(x.data_ptr(), y.data_ptr(), n, mn, mn + R, s.cuda_stream) == rtcdf.OK
    for seed in (7, 8):
        gen.keys_device(x.data_ptr(), n, mn, R, gen.UNIFORM, seed, stream=stream_handle())
        g.replay()
        torch.cuda.synchronize()
        assert_matches_oracle(x, y, mn, mn + R)


@pytest.mark.parametrize("key", [-1, 1_000_000, 1_000_000 + (1 << 15), np.iinfo(np.int32).max, np.iinfo(np.int32).min])
def test_partitioned_histogram_reports_a_key_out_of_range(key):
    n, R = 4_000_000, 1_000_000
    x = dev_keys(n, 0, R, gen.UNIFORM, 9)
    x[n // 2 + 1] = int(key)
    out = torch.empty_like(x)
    assert rtcdf.rtcdf_sort(x.data_ptr(), out.data_ptr(), n, 0, R, stream_handle()) == rtcdf.OK
    rc, bits = rtcdf.rtcdf_status_get(stream_handle())
    assert rc == rtcdf.ERR_KEY_OUT_OF_RANGE and bits == rtcdf.DEV_KEY_OUT_OF_RANGE
    x[n // 2 + 1] = 3
    gpu_sort(x, 0, R, out)
    assert_matches_oracle(x, out, 0, R)


# One scan CTA per 4096 values up to two per SM (304 on GB300), several chunks
# each beyond: both sides of the step, a last chunk of one value.
@pytest.mark.parametrize("R", [304 * 4096, 304 * 4096 + 1, 305 * 4096, 3 * 304 * 4096 + 17])
@pytest.mark.parametrize("dist", [gen.UNIFORM, gen.ALL_EQUAL])
def test_windows_over_a_wide_range(R, dist):
    n, mn, s = 700_001, -3, stream_handle()
    x = dev_keys(n, mn, R, dist, gen.derive_seed(33, R))
    counts = torch.zeros(R, dtype=torch.int32, device="cuda")
    assert rtcdf.rtcdf_hist_accumulate(x.data_ptr(), n, mn, mn + R, counts.data_ptr(), s) == rtcdf.OK
    wsb = rtcdf.rtcdf_workspace_size(R)
    ws = torch.zeros(wsb // 4, dtype=torch.int32, device="cuda")
    out = torch.empty_like(x)
    for lo, hi in ((0, 1), (1, 300_002), (300_002, n)):
        assert rtcdf.rtcdf_fill_from_counts(counts.data_ptr(), n, mn, mn + R, lo, hi, out.data_ptr() + 4 * lo,
                                            ws.data_ptr(), wsb, s) == rtcdf.OK
    assert rtcdf.rtcdf_ws_status_get(ws.data_ptr(), s) == (rtcdf.OK, 0)
    assert_matches_oracle(x, out, mn, mn + R)


def test_nothing_is_written_while_a_timeout_is_unread():
    n, R = 4_000_000, 1 << 20
    x = dev_keys(n, 0, R, gen.UNIFORM, 10)
    out = torch.full_like(x, -7)
    wsb = rtcdf.rtcdf_workspace_size(R)
    ws = torch.zeros(wsb // 4, dtype=torch.int32, device="cuda")
    ws[0] = rtcdf.DEV_TIMEOUT                    # control block word 0: the status
    s = stream_handle()
    assert rtcdf.rtcdf_sort_ws(x.data_ptr(), out.data_ptr(), n, 0, R, ws.data_ptr(), wsb, s) == rtcdf.OK
    assert rtcdf.rtcdf_ws_status_get(ws.data_ptr(), s)[0] == rtcdf.ERR_TIMEOUT
    assert bool((out == -7).all())
    assert rtcdf.rtcdf_sort_ws(x.data_ptr(), out.data_ptr(), n, 0, R, ws.data_ptr(), wsb, s) == rtcdf.OK
    assert rtcdf.rtcdf_ws_status_get(ws.data_ptr(), s) == (rtcdf.OK, 0)
    assert_matches_oracle(x, out, 0, R)


# Output of short runs: few keys per value, up to the step at 256, values present
# now and then, and outputs at every alignment.
@pytest.mark.parametrize("R,n", [(4096, 4096 * 256 - 1), (4096, 4096 * 256), (5000, 20_011), (50_000, 3), (300_000, 1_000_003),
                                 (1 << 22, 100_000), (1 << 22, 6_000_001)])
@pytest.mark.parametrize("dist", [gen.UNIFORM, gen.NORMAL])
@pytest.mark.parametrize("offset", [0, 1, 2, 3])
def test_short_runs(R, n, dist, offset):
    mn = -(1 << 31)                # the value that marks no run wraps around
    x = dev_keys(n, mn, R, dist, gen.derive_seed(35, R, n))
    out = torch.full((n + 8,), 5, dtype=torch.int32, device="cuda")
    gpu_sort(x, mn, mn + R, out[offset:offset + n])
    assert_matches_oracle(x, out[offset:offset + n], mn, mn + R)
    assert bool((out[:offset] == 5).all()) and bool((out[offset + n:] == 5).all())


def _wide_shape(name, n, R):
    g = torch.Generator("cuda")
    g.manual_seed(R)
    x = (torch.rand(n, device="cuda", generator=g, dtype=torch.float64) * R).int().clamp_(0, R - 1)
    if name == "half":             # half of a tile's values: the most that its table leaves the others out for
        x = x // 2 * 2
    elif name == "one":
        x.fill_(R - 1)
    elif name == "ends":           # the first and last value of every tile, and long runs
        x = (x // 16384 * 16384 + torch.where(x % 2 == 0, 0, 16383)).clamp_(max=R - 1)
    elif name == "gap":            # a long run and a few keys: most tiles empty
        x = torch.where(x % 1000 == 0, x, R // 3)
    return x.int()


# Scan and output in one launch: the narrowest and widest range, tiles of 16384
# values with a last one of a single value, whole and absent, the most keys a
# value and one more, few keys; against the oracle and against the launches of
# the general path (which explicit parameters select).
@pytest.mark.parametrize("R,n", [(999_999, 3_000_001), (1_000_000, 20_000_000), (1_000_000, 20_000_001), (31 * 32768 + 1, 2_800_002),
                                 (31 * 32768 + 16384, 2_900_003), (31 * 32768 + 16385, 2_900_001), (1 << 22, 5_000_002),
                                 (1 << 24, 200_003), (1 << 24, 30_000_001)])
@pytest.mark.parametrize("shape", ["uniform", "half", "one", "ends", "gap"])
def test_scan_and_output_of_a_wide_range(R, n, shape):
    mn, k = -(1 << 31), n % 4
    x = _wide_shape(shape, n, R) + mn
    out = torch.full((n + 8,), 5, dtype=torch.int32, device="cuda")
    gpu_sort(x, mn, mn + R, out[k:k + n])
    assert_matches_oracle(x, out[k:k + n], mn, mn + R)
    assert bool((out[:k] == 5).all()) and bool((out[k + n:] == 5).all())
    s, wsb = stream_handle(), rtcdf.rtcdf_workspace_size(R)
    ws = torch.zeros(wsb // 4, dtype=torch.int32, device="cuda")
    general = torch.empty_like(x)
    for params, dst in ((rtcdf.Params(), general), (None, out[k:k + n]), (rtcdf.Params(), general)):
        dst.fill_(0)               # one workspace for both, in turn
        assert rtcdf.rtcdf_sort_ex(x.data_ptr(), dst.data_ptr(), n, mn, mn + R, params, ws.data_ptr(), wsb, None, s) == rtcdf.OK
    assert rtcdf.rtcdf_ws_status_get(ws.data_ptr(), s) == (rtcdf.OK, 0)
    assert torch.equal(general, out[k:k + n])


# Keys past the last value: in its tile, in the bucket's other half, beyond.
@pytest.mark.parametrize("R", [31 * 32768 + 7, 31 * 32768 + 16384, 31 * 32768 + 20_000, 31 * 32768])
@pytest.mark.parametrize("past", [0, 16_383, 16_384, 40_000])
def test_wide_output_reports_a_key_past_the_range(R, past):
    n, s = 3_000_000, stream_handle()
    x = dev_keys(n, 0, R, gen.UNIFORM, 14)
    x[17] = R + past
    out = torch.empty_like(x)
    assert rtcdf.rtcdf_sort(x.data_ptr(), out.data_ptr(), n, 0, R, s) == rtcdf.OK
    assert rtcdf.rtcdf_status_get(s) == (rtcdf.ERR_KEY_OUT_OF_RANGE, rtcdf.DEV_KEY_OUT_OF_RANGE)
    want = torch.cat([x[:17], x[18:]]).sort().values
    assert torch.equal(out[:n - 1], want)
    x[17] = 0
    gpu_sort(x, 0, R, out)
    assert_matches_oracle(x, out, 0, R)


def test_wide_output_reports_a_stray_ticket():
    n, R, s = 300_000, 1 << 24, stream_handle()  # (more tiles than CTAs)
    x = dev_keys(n, 0, R, gen.UNIFORM, 15)
    out = torch.empty_like(x)
    wsb = rtcdf.rtcdf_workspace_size(R)
    ws = torch.zeros(wsb // 4, dtype=torch.int32, device="cuda")
    ws[1] = 2                      # control block word 1: the scan's ticket
    assert rtcdf.rtcdf_sort_ws(x.data_ptr(), out.data_ptr(), n, 0, R, ws.data_ptr(), wsb, s) == rtcdf.OK
    assert rtcdf.rtcdf_ws_status_get(ws.data_ptr(), s) == (rtcdf.ERR_TIMEOUT, rtcdf.DEV_TIMEOUT)
    ws.zero_()
    assert rtcdf.rtcdf_sort_ws(x.data_ptr(), out.data_ptr(), n, 0, R, ws.data_ptr(), wsb, s) == rtcdf.OK
    assert rtcdf.rtcdf_ws_status_get(ws.data_ptr(), s) == (rtcdf.OK, 0)
    assert_matches_oracle(x, out, 0, R)


# Few keys over a wide range: the fewest that the output buffer holds the partition
# of and fewer, both sides of the keys from which 2^20 < R < 2^22 is partitioned.
@pytest.mark.parametrize("R,n", [(1 << 22, 100), (1 << 22, 2600), (1 << 22, 2774), (1 << 22, 3001), ((1 << 22) + 1, 5003),
                                 (1 << 24, 16_000), (1 << 24, 30_001), (1_000_000, 1_538_461), (1_000_000, 1_538_462),
                                 (1 << 21, 625_000), (1 << 21, 625_001)])
@pytest.mark.parametrize("dist", [gen.UNIFORM, gen.NORMAL, gen.ALL_EQUAL])
def test_few_keys_over_a_wide_range(R, n, dist):
    mn = (1 << 31) - R
    for k in range(4):
        x = torch.empty(n + 3, dtype=torch.int32, device="cuda")[k:k + n]
        gen.keys_device(x.data_ptr(), n, mn, R, dist, gen.derive_seed(36, R, n, k), stream=stream_handle())
        out = torch.full((n + 8,), 5, dtype=torch.int32, device="cuda")
        gpu_sort(x, mn, mn + R, out[3 - k:3 - k + n])
        assert_matches_oracle(x, out[3 - k:3 - k + n], mn, mn + R)
        assert bool((out[:3 - k] == 5).all()) and bool((out[3 - k + n:] == 5).all())
