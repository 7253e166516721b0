"""The packed histogram (ranges of a few shared-memory tiles, many keys) where its
form changes and where its counters overflow: against the CPU oracle."""
import numpy as np
import pytest
import torch

import oracle
from gpu_util import assert_matches_oracle, dev_keys, gpu_sort, stream_handle
from paper_2609_00843_gb300 import gen, rtcdf

pytestmark = pytest.mark.gpu


# Both ends of every layout (2, 4, 5, 6, 8 fields a word) and of the whole range,
# just enough keys, with and without keys outside whole vectors.
@pytest.mark.parametrize("R,n,offset", [
    (49153, 36_000_001, 1), (65536, 35_000_002, 0), (65537, 36_000_003, 3), (131072, 24_000_000, 2),
    (131073, 24_000_001, 0), (163841, 24_000_002, 1), (270336, 14_000_001, 0), (270337, 14_000_002, 3),
    (360448, 10_000_003, 0), (360449, 10_000_000, 1),
])
@pytest.mark.parametrize("dist", [gen.UNIFORM, gen.NORMAL, gen.ALL_EQUAL])
def test_packed_histogram(R, n, offset, dist):
    mn = (1 << 31) - R if dist == gen.NORMAL else -7
    x = torch.empty(n + offset, dtype=torch.int32, device="cuda")[offset:]
    gen.keys_device(x.data_ptr(), n, mn, R, dist, gen.derive_seed(41, R), stream=stream_handle())
    out = torch.full((n + 3,), 77, dtype=torch.int32, device="cuda")[3 - offset:3 - offset + n]
    gpu_sort(x, mn, mn + R, out)
    assert_matches_oracle(x, out, mn, mn + R)


def _shape(name, n, R):
    g = torch.Generator("cuda")
    g.manual_seed(n)
    u = torch.rand(n, device="cuda", generator=g)
    x = (torch.rand(n, device="cuda", generator=g, dtype=torch.float64) * R).int().clamp_(0, R - 1)
    if name == "overflow":         # five keys of 0.08 % each: too rare for the sample, too many for a field
        x = torch.where(u < 0.004, (u * 1250).int() * 1000 + 11, x)
    elif name == "hot":            # one key of 90 %
        x = torch.where(u < 0.9, R // 2, x)
    elif name == "two":
        x = torch.where(u < 0.5, 3, R - 1)
    elif name == "multiples":
        x = x // 64 * 64
    elif name == "sorted":
        x = x.sort().values
    return x.int()


@pytest.mark.parametrize("R,n", [(65536, 40_000_001), (131072, 30_000_000), (1 << 18, 20_000_003), (350_000, 50_000_000)])
@pytest.mark.parametrize("shape", ["overflow", "hot", "two", "multiples", "sorted"])
def test_packed_histogram_of_uneven_keys(R, n, shape):
    x = _shape(shape, n, R)
    assert_matches_oracle(x, gpu_sort(x, 0, R), 0, R)


def test_packed_histogram_in_several_rounds():
    n, R = 60_000_001, 350_000     # 4-bit fields: about 4 keys of a CTA in the fullest
    x = dev_keys(n, 0, R, gen.NORMAL, 12)
    assert_matches_oracle(x, gpu_sort(x, 0, R), 0, R)


@pytest.mark.parametrize("shape", ["uniform", "overflow", "hot", "sorted"])
def test_packed_counts_add_up_without_scratch(shape):
    n, R, s = 30_000_001, 1 << 18, stream_handle()
    x = _shape(shape, n, R)
    counts = torch.zeros(R, dtype=torch.int32, device="cuda")
    for _ in range(2):
        assert rtcdf.rtcdf_hist_accumulate(x.data_ptr(), n, 0, R, counts.data_ptr(), s) == rtcdf.OK
    want = 2 * np.bincount(x.cpu().numpy(), minlength=R)
    assert np.array_equal(counts.cpu().numpy(), want)
    y = x.clone()
    gpu_sort(y, 0, R, y)           # in place: no scratch either
    assert np.array_equal(y.cpu().numpy(), oracle.counting_sort(x.cpu().numpy(), 0, R))


@pytest.mark.parametrize("key", [-1, 200_000, np.iinfo(np.int32).max, np.iinfo(np.int32).min])
def test_packed_histogram_reports_a_key_out_of_range(key):
    n, R = 20_000_000, 200_000
    x = dev_keys(n, 0, R, gen.UNIFORM, 13)
    x[n - 5] = int(key)
    out = torch.empty_like(x)
    assert rtcdf.rtcdf_sort(x.data_ptr(), out.data_ptr(), n, 0, R, stream_handle()) == rtcdf.OK
    rc, bits = rtcdf.rtcdf_status_get(stream_handle())
    assert rc == rtcdf.ERR_KEY_OUT_OF_RANGE and bits == rtcdf.DEV_KEY_OUT_OF_RANGE
    x[n - 5] = 3
    gpu_sort(x, 0, R, out)
    assert_matches_oracle(x, out, 0, R)


# Pairs of CTAs add up their fields: every layout, and several rounds (normal keys).
@pytest.mark.parametrize("R,n", [(49153, 45_000_001), (131071, 28_000_002), (163840, 21_000_003), (270336, 14_000_001),
                                 (350_001, 60_000_000)])
@pytest.mark.parametrize("dist", [gen.UNIFORM, gen.NORMAL])
def test_packed_counts_of_every_layout_without_scratch(R, n, dist):
    x = dev_keys(n, -5, R, dist, R)
    counts = torch.zeros(R, dtype=torch.int32, device="cuda")
    assert rtcdf.rtcdf_hist_accumulate(x.data_ptr(), n, -5, R - 5, counts.data_ptr(), stream_handle()) == rtcdf.OK
    assert np.array_equal(counts.cpu().numpy(), np.bincount(x.cpu().numpy() + 5, minlength=R))


def test_nothing_is_written_while_a_timeout_is_unread():
    n, R, s = 20_000_000, 1 << 18, stream_handle()
    x = dev_keys(n, 0, R, gen.UNIFORM, 16)
    out = torch.full_like(x, -7)
    wsb = rtcdf.rtcdf_workspace_size(R)
    ws = torch.zeros(wsb // 4, dtype=torch.int32, device="cuda")
    ws[0] = rtcdf.DEV_TIMEOUT                    # control block word 0: the status
    assert rtcdf.rtcdf_sort_ws(x.data_ptr(), out.data_ptr(), n, 0, R, ws.data_ptr(), wsb, s) == rtcdf.OK
    assert rtcdf.rtcdf_ws_status_get(ws.data_ptr(), s)[0] == rtcdf.ERR_TIMEOUT
    assert bool((out == -7).all())
    assert rtcdf.rtcdf_sort_ws(x.data_ptr(), out.data_ptr(), n, 0, R, ws.data_ptr(), wsb, s) == rtcdf.OK
    assert rtcdf.rtcdf_ws_status_get(ws.data_ptr(), s) == (rtcdf.OK, 0)
    assert_matches_oracle(x, out, 0, R)
