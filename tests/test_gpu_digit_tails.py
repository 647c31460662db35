"""Digit sorts (csrc/radix.cu) whose last tile is partial, against the oracle:
1 to 15 keys past a step of the ranking, where keys and padding share one
atomic, with many keys whose digits are all ones up to the top one (i32 -1,
f32 -0.0) and so lie next to the padding, on each route.  Sorts are exact: no
tolerance."""
import numpy as np
import pytest

import oracle
from paper_2409_03970_gb300 import inputs

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

CLUSTER, PASSES = ["radix_cluster"], ["radix_histogram", "radix_pass"]


@pytest.fixture(scope="module")
def ns():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2409_03970_gb300 import build, nsort
    build.build()
    nsort.lib()
    return nsort


def near_padding(n, dt, seed):
    """A third each: the key next to the padding, keys with some digits of
    all ones, uniform keys."""
    wide = dt in inputs.KEY64_DTYPES
    x = inputs.keys64(n, "u64", "uniform", seed) if wide else inputs.keys(n, "u32", "uniform", seed)
    pick = inputs.counter_u32(seed, 3, 0, n)
    ones = np.array(-1, x.dtype.str.replace("u", "i")).view(x.dtype)
    top = x.dtype.type(1 << (8 * x.dtype.itemsize - 1))
    shift = (8 * (pick >> 8 & (x.dtype.itemsize - 1))).astype(x.dtype)
    x = np.where(pick % 3 == 1, x | (ones >> shift), x)
    return np.where(pick % 3 == 0, top if dt in ("f32", "f64") else ones, x)


# (route, sizes are these plus 1 .. 15): clusters of 4 to 16 keys a thread, wave
# passes in clusters of four, of one large and of one small tile, look-back passes
SIZES32 = [(CLUSTER, 16384), (CLUSTER, 40_000), (CLUSTER, 120_000), (PASSES, 200_000),
           (PASSES, 1_700_000), (PASSES, 2_600_000), (PASSES, 5_000_000)]
SIZES64 = [(PASSES, 700_000), (PASSES, 1_200_000), (PASSES, 1_500_000), (PASSES, 2_600_000)]


@pytest.mark.parametrize("dt,code", [("i32", 1), ("f32", 2), ("i64", 4), ("f64", 5)])
def test_tails(ns, dt, code):
    wide = dt in inputs.KEY64_DTYPES
    for want_route, base in SIZES64 if wide else SIZES32:
        big = near_padding(base + 15, dt, base)
        tmp = ns.scratch(ns.KIND_KEYS, big.size, dtype=code)
        for n in range(base // 16 * 16 + 1, base // 16 * 16 + 16):
            bits = big[-n:]
            x = torch.from_numpy(bits.view(np.int64 if wide else np.int32).copy()).cuda()
            out = torch.empty_like(x)
            ns.nsort_trace_enable(True)
            assert ns.nsort_keys(x, out, n, code, tmp, tmp.numel()) == ns.OK
            assert ns.nsort_device_status(tmp) == ns.OK
            trace = ns.nsort_trace_read()
            ns.nsort_trace_enable(False)
            assert sorted(k for k in trace if k.startswith(("radix", "merge"))) == want_route, n
            want = oracle.sort_keys64(bits, dt) if wide else oracle.sort_keys(bits, dt)
            np.testing.assert_array_equal(out.cpu().numpy().view(bits.dtype), want, err_msg=f"{n}")
