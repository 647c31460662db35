"""The digit sorts of arrays beyond one tile (csrc/radix.cu) against the
oracle, bit for bit, at the sizes where the route changes (one cluster of 16
CTAs, passes of tiles that all run at once, look-back passes) and at the edges
of their tiles; distributions for each way of ranking (keys that agree in the
sorted digits, keys that do not, a mix, one digit for a whole tile), keys
equal to the padding of the last tile, in place, and buffers of any
alignment.  Sorts are exact: no tolerance."""
import numpy as np
import pytest

import oracle
from paper_2409_03970_gb300 import inputs

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

CODE = {"u32": 0, "i32": 1, "f32": 2, "u64": 3, "i64": 4, "f64": 5}


@pytest.fixture(scope="module")
def ns():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2409_03970_gb300 import build, nsort
    build.build()
    nsort.lib()
    return nsort


def cuda(a, offset=0):
    """A device copy of a that starts `offset` elements past an allocation."""
    t = {4: torch.int32, 8: torch.int64}[a.dtype.itemsize]
    x = torch.empty(a.size + offset, dtype=t, device="cuda")
    x[offset:] = torch.from_numpy(a.view({4: np.int32, 8: np.int64}[a.dtype.itemsize]))
    return x[offset:]


def draw(n, dt, dist, seed):
    if dt in inputs.KEY64_DTYPES:
        if dist == "ones":
            return np.full(n, 2**64 - 1, np.uint64)
        if dist == "low":      # small numbers: the upper digits are all alike
            return inputs.keys64(n, "u64", "uniform", seed) >> np.uint64(50)
        return inputs.keys64(n, dt, dist, seed)
    if dist == "ones":         # the key that pads the last tile
        return np.full(n, 2**32 - 1, np.uint32)
    if dist == "low":
        return inputs.keys(n, "u32", "uniform", seed) >> np.uint32(20)
    return inputs.keys(n, dt, dist, seed)


def run(ns, kind, dt, keys, vals, inplace=False, offset=0):
    n = keys.size
    k = cuda(keys, offset)
    ko = k if inplace else torch.empty(n + offset, dtype=k.dtype, device="cuda")[offset:]
    v = vo = None
    if vals is not None:
        v = cuda(vals, offset)
        vo = v if inplace else torch.empty(n + offset, dtype=v.dtype, device="cuda")[offset:]
    need = ns.nsort_temp_bytes(kind, n, 0, CODE[dt])
    tmp = torch.full((need + 256,), 0x5A, dtype=torch.uint8, device="cuda")   # any contents
    ns.nsort_trace_enable(True)
    if kind == ns.KIND_KEYS:
        rc = ns.nsort_keys(k, ko, n, CODE[dt], tmp, need)
    elif kind == ns.KIND_PAIRS:
        rc = ns.nsort_pairs(k, v, ko, vo, n, CODE[dt], tmp, need)
    else:
        rc = ns.nsort_pairs64(k, v, ko, vo, n, CODE[dt], tmp, need)
    assert rc == ns.OK, ns.lib().nsort_last_error()
    assert ns.nsort_device_status(tmp) == ns.OK
    trace = ns.nsort_trace_read()
    ns.nsort_trace_enable(False)
    assert bool((tmp[need:] == 0x5A).all()), "wrote past the scratch"
    route = sorted(k for k in trace if k.startswith("radix") or k.startswith("merge"))
    if "radix_pass" in trace:
        assert trace["radix_pass"]["launches"] == keys.dtype.itemsize
    out = [x.cpu().numpy().view(keys.dtype if i == 0 else vals.dtype)
           for i, x in enumerate([ko] + ([] if vo is None else [vo]))]
    return route, out


CLUSTER, PASSES = ["radix_cluster"], ["radix_histogram", "radix_pass"]
DISTS = ["uniform", "sorted", "dup16", "zipf", "low", "ones"]


def sizes32(merge_tile):
    """(n, route) of 32-bit keys and pairs: one cluster from two sort tiles
    on, passes while 2 CTAs per SM hold all tiles, then look-back passes."""
    at_once = 2 * torch.cuda.get_device_properties(0).multi_processor_count
    clusters = (at_once // 4) * 4 * 4096
    return [(merge_tile + 1, CLUSTER), (32768, CLUSTER), (32769, CLUSTER), (65536, CLUSTER),
            (65537, None), (131072, None), (131073, None), (200_003, PASSES),
            (clusters, PASSES), (clusters + 1, PASSES), (at_once // 2 * 10240 + 1, PASSES),
            (at_once // 2 * 16384, PASSES), (at_once // 2 * 16384 + 1, PASSES),
            (at_once * 10240 + 1, PASSES), (at_once * 16384 + 1, PASSES)]


def sizes64():
    at_once = 2 * torch.cuda.get_device_properties(0).multi_processor_count
    return [((5 << 17) - 1, ["merge_keys64"]), (5 << 17, PASSES),
            (at_once // 2 * 6144, PASSES), (at_once // 2 * 6144 + 1, ["merge_keys64"]),
            ((9 << 17) - 1, ["merge_keys64"]), (9 << 17, PASSES), (at_once // 2 * 8192, PASSES),
            (at_once // 2 * 8192 + 1, PASSES), (at_once * 6144 + 1, PASSES),
            (at_once * 8192, PASSES), (at_once * 8192 + 1, PASSES), ((1 << 22) - 1, PASSES)]


@pytest.mark.parametrize("dt", ["u32", "i32", "f32", "i64", "f64"])
def test_keys(ns, dt):
    wide = dt in inputs.KEY64_DTYPES
    for i, (n, want_route) in enumerate(sizes64() if wide else sizes32(16384)):
        for dist in DISTS:
            if wide and dist == "zipf" or (n > 3_000_000 and dist in ("sorted", "low")):
                continue
            x = draw(n, dt, dist, seed=n)
            want = oracle.sort_keys64(x, dt) if wide else oracle.sort_keys(x, dt)
            route, (got,) = run(ns, ns.KIND_KEYS, dt, x, None, inplace=i % 2 == 1, offset=i % 3)
            assert want_route is None or route == want_route
            np.testing.assert_array_equal(got, want, err_msg=f"{n} {dist}")


@pytest.mark.parametrize("vbytes", [4, 8])
def test_pairs(ns, vbytes):
    kind = ns.KIND_PAIRS if vbytes == 4 else ns.KIND_PAIRS64
    for i, (n, want_route) in enumerate(sizes32(8192)):
        # (pairs64 takes 16-byte aligned outputs only)
        offset = (i % 3) if vbytes == 4 else 0
        for dist in DISTS:
            if n > 3_000_000 and dist in ("sorted", "low"):
                continue
            dt = ["f32", "i32", "u32"][i % 3]
            x = draw(n, dt, dist, seed=n)
            order = np.arange(n, dtype=np.uint32)
            wk, perm = oracle.sort_pairs(x, order, dt)
            v = order if vbytes == 4 else inputs.counter_u64(n, 7, 0, n)
            route, (gk, gv) = run(ns, kind, dt, x, v, inplace=i % 2 == 1, offset=offset)
            assert want_route is None or route == want_route
            np.testing.assert_array_equal(gk, wk, err_msg=f"{n} {dist}")
            np.testing.assert_array_equal(gv, v[perm], err_msg=f"{n} {dist}")
