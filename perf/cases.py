"""Performance cases of the RT-CDF sort: what a user's program has it do.

Every case goes through the public Python binding (``rtcdf.sort``,
``BatchPlan``, ``rtcdf_sort_batched_device_ws``, ``rtcdf_sort_host``,
``dist.ShardedSorter``) with seeded inputs in the shapes of the paper's
evaluation (uniform, normal, one value).  A case's ``kind`` says which call it
makes; the remaining fields are its sizes.
"""
import math

import numpy as np
import torch

from paper_2609_00843_gb300 import dist, gen, rtcdf

# "constant": one value, after up to 1000 keys of another one.
SHAPES = ("uniform", "normal", "constant")

# Ranges that drawn cases come from (both ends reached).
N_RANGE = (10_000, 100_000_000)      # keys of one device array
R_RANGE = (2, 1 << 24)               # values of its range; the library's limit is 2^24
HOST_N_RANGE = (100_000, 20_000_000)
SHARD_N_RANGE = (1_000_000, 50_000_000)
SEG_RANGE = (64, 4096)               # segments; each 1e3..1e6 keys over 2^7..2^16 values


def listed():
    return [
        # The smallest requests of a sort service: latency and launches only.
        dict(name="tiny_1e4_r1000", kind="sort", n=10_007, minVal=0, R=1000, shape="normal", offset=0),
        # One small column of byte-like codes, sorted on its own.
        dict(name="small_1e6_r128", kind="sort", n=1_000_000, minVal=0, R=128, shape="uniform", offset=0),
        # A slice of a larger buffer: odd length, not 16-byte aligned, odd range.
        dict(name="ragged_3e6_r50021", kind="sort", n=3_141_593, minVal=-70_001, R=50_021, shape="normal",
             offset=1),
        # A large column whose range fits one shared-memory histogram.
        dict(name="column_1e8_r2e14", kind="sort", n=100_000_000, minVal=-1000, R=1 << 14, shape="uniform",
             offset=0),
        # A large column of 18-bit keys (ids, quantised measurements), peaked.
        dict(name="column_1e8_r2e18", kind="sort", n=100_000_000, minVal=-1000, R=1 << 18, shape="normal",
             offset=0),
        # The largest array: 4 GB of 16-bit keys.
        dict(name="large_1e9_r2e16", kind="sort", n=1_000_000_000, minVal=0, R=1 << 16, shape="normal", offset=0),
        # Wide ranges: 20-bit ids over an odd range, and the widest range the library takes.
        dict(name="wide_3e7_r1e6", kind="sort", n=30_000_001, minVal=-500_000, R=1_000_003, shape="uniform",
             offset=0),
        dict(name="widest_1e8_r2e24", kind="sort", n=100_000_000, minVal=-(1 << 23), R=1 << 24, shape="normal",
             offset=0),
        # Many groups sorted at once, the same layout again and again (a plan kept by the program).
        dict(name="segments_4096_plan", kind="plan", segments=4096, layout=3),
        # Groups whose layout only the device knows, planned on the device.
        dict(name="segments_1024_device", kind="device", segments=1024, layout=5),
        # Keys in page-locked host memory, sorted through the device.
        dict(name="host_2e7_r4096", kind="host", n=20_000_000, minVal=0, R=4096, shape="uniform"),
        # One rank's share of a sharded array: counts, exchange, its window.
        dict(name="shard_5e7_r2e18", kind="shard", n=50_000_000, minVal=0, R=1 << 18, shape="uniform"),
    ]


def _log_int(rng, lo, hi):
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    kind = rng.choice(("sort", "sort", "sort", "sort", "plan", "device", "host", "shard"))
    if kind in ("plan", "device"):
        return dict(kind=kind, segments=_log_int(rng, *SEG_RANGE), layout=rng.randrange(1, 1 << 20))
    case = dict(kind=kind, R=_log_int(rng, *R_RANGE), shape=rng.choice(SHAPES))
    case["minVal"] = rng.randrange(-(1 << 24), 1 << 24)
    if kind == "sort":
        case.update(n=_log_int(rng, *N_RANGE), offset=rng.randrange(4))
    elif kind == "host":
        case.update(n=_log_int(rng, *HOST_N_RANGE))
    else:
        case.update(n=_log_int(rng, *SHARD_N_RANGE))
    return case


def _stream():
    return torch.cuda.current_stream().cuda_stream


def _keys(case, seed, offset=0):
    """The case's keys on the device, starting `offset` elements into their buffer."""
    n, R, mn = case["n"], case["R"], case["minVal"]
    sd = gen.derive_seed(seed, n, R)
    x = torch.empty(n + offset, dtype=torch.int32, device="cuda")[offset:]
    if case["shape"] == "constant":
        x.fill_(mn + sd % R)
        x[:1 + (sd >> 32) % 1000] = mn + (sd + 1) % R
    else:
        gen.keys_device(x.data_ptr(), n, mn, R, gen.DIST_NAMES[case["shape"]], sd, stream=_stream())
    return x


def _layout(case):
    """Offsets, minVal, maxVal and shape of the segments: the layout does not
    depend on the inputs' seed."""
    n, mn, R, shape, _ = gen.batched_segments(gen.derive_seed(case["layout"]), case["segments"])
    offs = np.zeros(case["segments"] + 1, np.int64)
    offs[1:] = np.cumsum(n)
    return offs, mn, mn + R, shape


def _segment_keys(offs, mn, mx, shape, seed):
    x = torch.empty(int(offs[-1]), dtype=torch.int32, device="cuda")
    for i in range(len(mn)):
        lo, hi = int(offs[i]), int(offs[i + 1])
        gen.keys_device(x.data_ptr() + 4 * lo, hi - lo, int(mn[i]), int(mx[i] - mn[i]), int(shape[i]),
                        gen.derive_seed(seed, i), stream=_stream())
    return x


def prepare(case, seed):
    kind = case["kind"]
    st = dict(kind=kind)
    if kind in ("plan", "device"):
        offs, mn, mx, shape = _layout(case)
        st["x"] = _segment_keys(offs, mn, mx, shape, seed)
        st["out"] = torch.empty_like(st["x"])
        if kind == "plan":
            st["plan"] = rtcdf.BatchPlan(offs, mn, mx)
            st["ws"] = torch.zeros(st["plan"].workspace_size(), dtype=torch.uint8, device="cuda")
        else:
            st["meta"] = [torch.from_numpy(a).cuda() for a in (offs, mn, mx)]
            st["bounds"] = len(mn), int(offs[-1]), int((mx - mn).max())
            st["ws"] = torch.zeros(rtcdf.rtcdf_batch_device_workspace_size(*st["bounds"]), dtype=torch.uint8,
                                   device="cuda")
        return st
    st["minVal"], st["maxVal"] = case["minVal"], case["minVal"] + case["R"]
    st["x"] = _keys(case, seed, case.get("offset", 0))
    if kind == "host":
        st["x"] = st["x"].cpu().pin_memory()
        st["out"] = torch.empty_like(st["x"]).pin_memory()
    else:
        st["out"] = torch.empty_like(st["x"])
    if kind == "shard":
        st["sorter"] = dist.ShardedSorter(case["R"])
    return st


def run(state):
    x, out, kind = state["x"], state["out"], state["kind"]
    if kind == "sort":
        return rtcdf.sort(x, state["minVal"], state["maxVal"], out=out)
    if kind == "shard":
        return state["sorter"].sort(x, x.numel(), state["minVal"], state["maxVal"], out)
    if kind == "plan":
        rc = state["plan"].run(x.data_ptr(), out.data_ptr(), state["ws"].data_ptr(), state["ws"].numel(), _stream())
    elif kind == "device":
        offs, mn, mx = state["meta"]
        rc = rtcdf.rtcdf_sort_batched_device_ws(x.data_ptr(), out.data_ptr(), offs.data_ptr(), mn.data_ptr(),
                                                mx.data_ptr(), *state["bounds"], state["ws"].data_ptr(),
                                                state["ws"].numel(), _stream())
    else:
        rc = rtcdf.rtcdf_sort_host(x.data_ptr(), out.data_ptr(), x.numel(), state["minVal"], state["maxVal"],
                                   _stream())
        torch.cuda.current_stream().synchronize()  # the program reads the result on the host
    if rc != rtcdf.OK:
        raise rtcdf.RtcdfError(rc, kind)
    return out


def work(case):
    """Each key read once and written once, and counted once."""
    n = int(_layout(case)[0][-1]) if case["kind"] in ("plan", "device") else case["n"]
    return {"bytes": 8 * n, "flops": n}


def exact(case, seed):
    if case["kind"] in ("plan", "device"):
        offs, mn, mx, shape = _layout(case)
        x = _segment_keys(offs, mn, mx, shape, seed).long()
        seg = torch.repeat_interleave(torch.arange(len(mn), device="cuda"),
                                      torch.from_numpy(np.diff(offs)).cuda())
        key = (seg << 32) | (x + (1 << 31))  # segment first, then the key shifted to be nonnegative
        return ((key.sort().values & 0xFFFFFFFF) - (1 << 31)).int()
    if case["n"] > 200_000_000:
        return None  # three 64-bit copies of the largest array take too long
    out = _keys(case, seed).long().sort().values.int()
    return out.cpu() if case["kind"] == "host" else out
