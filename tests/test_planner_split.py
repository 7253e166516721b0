"""Which in-CTA segments the device planner splits into work items: those that would
outlast the scan launch, unless so many are alike that splitting them costs more.  The
host emulation of the rule, and the planner kernel against it."""
import subprocess

import numpy as np
import pytest
import torch

from gpu_util import stream_handle
from paper_2609_00843_gb300 import rtcdf
from test_devplan_gpu import check_segments, emitter, make_layout, to_dev  # noqa: F401 (a fixture)


def equal(S, n, R):
    return [n] * S, [R] * S


def mixed(S, n_lo, n_hi, r_lo, r_hi, seed):
    g = np.random.default_rng(seed)
    draw = lambda lo, hi: np.exp(g.uniform(np.log(lo), np.log(hi), S)).astype(np.int64).tolist()  # noqa: E731
    return draw(n_lo, n_hi), draw(r_lo, r_hi)


def lists(exe, path, lengths, Rs, max_R=16000):
    """The lengths of the emulated plan's lists: n_first, n_scan, n_small2, ..."""
    offs = np.concatenate([[0], np.cumsum(lengths)])
    path.write_text(f"{len(lengths)} {offs[-1]} {max_R}\n" + " ".join(map(str, offs)) + "\n" +
                    " ".join(["0"] * len(lengths)) + "\n" + " ".join(map(str, Rs)) + "\n")
    r = subprocess.run([exe, "--emit", str(path)], capture_output=True, text=True, timeout=120)
    assert r.returncode == 0, r.stderr[-2000:]
    return [int(v) for v in next(ln for ln in r.stdout.splitlines() if ln.startswith("hdr")).split()[1:]]


# Few keys over a wide range, and many alike, are left whole; a few long ones, and the
# long ones of a mixed layout, are split.
@pytest.mark.parametrize("layout,split", [
    (equal(700, 1, 16000), 0), (equal(400, 2000, 16000), 0), (equal(8, 100, 16000), 0),
    (equal(400, 8000, 4000), 0), (equal(1024, 20_000, 16000), 0), (equal(256, 20_000, 128), 0),
    (equal(8, 20_000, 4000), 8), (equal(256, 60_000, 16000), 256), (equal(64, 20_000, 16000), 64),
])
def test_equal_segments(emitter, tmp_path, layout, split):  # noqa: F811
    S = len(layout[0])
    hdr = lists(emitter, tmp_path / "m", *layout)
    assert hdr[2] == S - split and (hdr[4] > 0) == (split > 0)


def test_long_segments_of_a_mixed_layout(emitter, tmp_path):  # noqa: F811
    L, R = mixed(500, 1e3, 6e4, 128, 16000, 3)
    outlast = sum(5000 + 21 * n // 20 + 19 * r // 10 > 21_000 and n > r // 8 for n, r in zip(L, R))
    hdr = lists(emitter, tmp_path / "m", L, R)
    assert 50 < outlast < 400 and hdr[2] == 500 - outlast


# 1024 segments are classified together: a block of equal ones beside a mixed one.
@pytest.mark.gpu
@pytest.mark.parametrize("layout", [
    equal(1, 60_000, 16000), equal(300, 8000, 4000),
    tuple(a + b for a, b in zip(mixed(1024, 1e3, 6e4, 128, 16000, 4), equal(900, 40_000, 8000))),
    tuple(a + b for a, b in zip(equal(1024, 50_000, 16000), mixed(3, 4e4, 6e4, 128, 16000, 5))),
])
def test_planner_kernel_splits_as_the_emulation(emitter, tmp_path, layout):  # noqa: F811
    L, R = layout
    hdr = lists(emitter, tmp_path / "m", L, R)
    x, offs, mn, mx = make_layout(L, R, [0] * len(L), [i % 2 for i in range(len(L))], range(len(L)))
    out = torch.empty_like(x)
    wsb, s = rtcdf.rtcdf_batch_device_workspace_size(len(L), x.numel(), 16000), stream_handle()
    ws = torch.zeros(wsb // 4, dtype=torch.int32, device="cuda")
    meta = [to_dev(v) for v in (offs, mn, mx)]
    for _ in range(2):
        assert rtcdf.rtcdf_sort_batched_device_ws(x.data_ptr(), out.data_ptr(), *[t.data_ptr() for t in meta], len(L),
                                                  x.numel(), 16000, ws.data_ptr(), wsb, s) == rtcdf.OK
        assert rtcdf.rtcdf_batch_status_get(ws.data_ptr(), s) == (rtcdf.OK, 0)
        assert ws[64:64 + 13].tolist() == hdr    # the header follows the control block
        check_segments(x, out, offs, mn, mx)
