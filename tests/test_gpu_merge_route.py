"""The plain sorts' merge passes, which 32-bit sorts take from 2^30 keys on only:
forced (nsort_testing_merge_sort) at the sizes where they find their splitters in
another way, on outputs off a 16-byte boundary, in place, against the four-way
passes; and the real calls on either side of 2^30.  Sorts are exact: no
tolerance."""
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


def kinds(ns):
    return {"keys": ns.KIND_KEYS, "pairs": ns.KIND_PAIRS, "pairs64": ns.KIND_PAIRS64}


def route(trace):
    return {k: v["launches"] for k, v in trace.items() if k.startswith(("radix", "merge"))}


def check(ns, op, dt, n, dist, inplace=False, offset=0):
    """One forced sort against the oracle, its passes against the plan."""
    kind, wide = kinds(ns)[op], dt in inputs.KEY64_DTYPES
    x = inputs.keys64(n, dt, dist, n) if wide else inputs.keys(n, dt, dist, n)
    word = torch.int64 if wide else torch.int32

    def dev(a, t):
        b = torch.empty(n + offset, dtype=t, device="cuda")
        b[offset:] = torch.from_numpy(a.view({torch.int32: np.int32, torch.int64: np.int64}[t]))
        return b[offset:]
    k = dev(x, word)
    ko = k if inplace else torch.empty(n + offset, dtype=word, device="cuda")[offset:]
    v = vo = None
    if op != "keys":
        vt = torch.int64 if op == "pairs64" else torch.int32
        payload = inputs.counter_u64(n, 7, 0, n) if op == "pairs64" else inputs.counter_u32(5, 6, 0, n)
        v = dev(payload, vt)
        vo = v if inplace else torch.empty(n + offset, dtype=vt, device="cuda")[offset:]
    tmp = ns.scratch(kind, n, dtype=CODE[dt])
    ns.nsort_trace_enable(True)
    assert ns.nsort_testing_merge_sort(kind, k, v, ko, vo, n, CODE[dt], tmp, tmp.numel()) == ns.OK
    assert ns.nsort_device_status(tmp) == ns.OK
    got = route(ns.nsort_trace_read())
    ns.nsort_trace_enable(False)
    passes = ns.nsort_plan(ns.KIND_KEYS if op == "keys" else ns.KIND_PAIRS, n, CODE[dt])[0] - 1
    assert got == {"merge_keys64" if wide else "merge_keys" if op == "keys" else "merge_pairs": passes}
    gk = ko.cpu().numpy().view(x.dtype)
    if op == "keys":
        want = oracle.sort_keys64(x, dt) if wide else oracle.sort_keys(x, dt)
        np.testing.assert_array_equal(gk, want)
        return
    wk, perm = oracle.sort_pairs(x, np.arange(n, dtype=np.uint32), dt)
    np.testing.assert_array_equal(gk, wk)
    np.testing.assert_array_equal(vo.cpu().numpy().view(payload.dtype), payload[perm])


def mode_size(ns, op, dt, point):
    """Sizes around one and two merge tiles per CTA of the last pass's grid."""
    grid = ns.nsort_merge_grid(ns.KIND_KEYS if op == "keys" else ns.KIND_PAIRS, CODE[dt])
    tile = ns.nsort_plan(ns.KIND_KEYS if op == "keys" else ns.KIND_PAIRS, 1 << 24, CODE[dt])[2]
    one, two = grid * tile, 2 * grid * tile
    return {"1x": one, "1x+1": one + 1, "1.5x": (one + two) // 2 + 17, "2x": two,
            "2x+1": two + 1, "2.1x": two + two // 20 + 11}[point]


@pytest.mark.parametrize("dist", ["uniform", "sorted", "dup16"])
@pytest.mark.parametrize("point", ["1x", "1x+1", "1.5x", "2x", "2x+1", "2.1x"])
@pytest.mark.parametrize("dt", ["f32", "i64"])
def test_keys_splitter_modes(ns, dt, point, dist):
    check(ns, "keys", dt, mode_size(ns, "keys", dt, point), dist)


@pytest.mark.parametrize("point", ["1x", "1x+1", "2x", "2x+1"])
@pytest.mark.parametrize("op", ["pairs", "pairs64"])
def test_pairs_splitter_modes(ns, op, point):
    check(ns, op, "i32", mode_size(ns, op, "i32", point), "dup16")


@pytest.mark.parametrize("n", [16385, 3 * 16384 + 7, 100_003, (1 << 20) + 12345])
@pytest.mark.parametrize("op,dt", [("keys", "u32"), ("keys", "f64"), ("pairs", "f32"), ("pairs64", "u32")])
def test_sizes_in_place_and_off_a_boundary(ns, op, dt, n):
    check(ns, op, dt, n, "uniform")
    check(ns, op, dt, n, "dup16", inplace=True)
    if op != "pairs64":                      # (takes 16-byte aligned outputs only)
        for offset in (1, 3):
            check(ns, op, dt, n, "dup16", offset=offset)


def test_two_way_and_four_way_agree(ns):
    n = (1 << 22) + 9
    bits, _ = inputs.normal_pairs(n, seed=7, special_per_mille=10)
    x = torch.from_numpy(bits.view(np.int32)).cuda()
    outs = []
    for setting, name in ((ns.FOUR_WAY_NEVER, "merge_keys"), (0, "merge4_keys")):
        prev = ns.nsort_testing_set_four_way_min(setting)
        try:
            need, out = ns.nsort_temp_bytes(ns.KIND_KEYS, n), torch.empty_like(x)
            tmp = torch.full((need + (1 << 17),), 0x5A, dtype=torch.uint8, device="cuda")
            ns.nsort_trace_enable(True)
            assert ns.nsort_testing_merge_sort(ns.KIND_KEYS, x, None, out, None, n, ns.F32, tmp,
                                               need) == ns.OK
            assert name in route(ns.nsort_trace_read())
            ns.nsort_trace_enable(False)
            assert ns.nsort_device_status(tmp) == ns.OK
            assert bool((tmp[need:] == 0x5A).all()), "wrote past the scratch"
        finally:
            ns.nsort_testing_set_four_way_min(prev)
        outs.append(out.cpu().numpy().view(np.uint32))
    np.testing.assert_array_equal(outs[0], oracle.sort_keys(bits, "f32"))
    np.testing.assert_array_equal(outs[0], outs[1])


def test_refuses_what_the_sorts_refuse(ns):
    n = 40_000
    x = torch.zeros(n, dtype=torch.int32, device="cuda")
    tmp = ns.scratch(ns.KIND_PAIRS64, n)
    call = ns.nsort_testing_merge_sort
    assert call(ns.KIND_KEYS, x, None, x, None, 16384, 0, tmp, tmp.numel()) == ns.EINVAL   # one tile
    assert call(ns.KIND_KEYS, x, None, x, None, n, 0, tmp, 1000) == ns.ENOMEM
    assert call(ns.KIND_PAIRS, x, None, x, None, n, 0, tmp, tmp.numel()) == ns.EINVAL
    assert call(ns.KIND_PAIRS64, x, x.data_ptr() + 4, x, x.data_ptr(), n, 0, tmp, tmp.numel()) == ns.EINVAL


@pytest.mark.parametrize("op,n", [("keys", (1 << 30) - 1), ("keys", 1 << 30), ("pairs", (1 << 30) - 1),
                                  ("pairs", 1 << 30), ("pairs64", 1 << 30)])
def test_on_either_side_of_2p30(ns, op, n):
    """The public calls: digits below 2^30 keys, merges from there on; payloads are
    positions, which give the input back, and rise among equal keys."""
    kind = kinds(ns)[op]
    g = torch.Generator(device="cuda")
    g.manual_seed(n)
    # (about four of each key, so that stability shows)
    x = torch.randint(-(1 << 27), 1 << 27, (n,), dtype=torch.int32, device="cuda", generator=g)
    out, tmp = torch.empty_like(x), ns.scratch(kind, n)
    ns.nsort_trace_enable(True)
    if op == "keys":
        assert ns.nsort_keys(x, out, n, ns.I32, tmp, tmp.numel()) == ns.OK
    else:
        v = torch.arange(n, dtype=torch.int64 if op == "pairs64" else torch.int32, device="cuda")
        vo = torch.empty_like(v)
        call = ns.nsort_pairs if op == "pairs" else ns.nsort_pairs64
        assert call(x, v, out, vo, n, ns.I32, tmp, tmp.numel()) == ns.OK
        del v
    assert ns.nsort_device_status(tmp) == ns.OK
    names = set(route(ns.nsort_trace_read()))
    ns.nsort_trace_enable(False)
    assert names == ({"radix_histogram", "radix_pass"} if n < 1 << 30 else
                     {"merge_keys" if op == "keys" else "merge_pairs"})
    del tmp
    assert bool((out[1:] >= out[:-1]).all())
    if op == "keys":          # the same keys: as many in each of 2^16 bands, the same sums of powers
        for f in (lambda t: t, lambda t: t * t, lambda t: t * t * t):
            assert int(f(x.long()).sum()) == int(f(out.long()).sum())
        assert torch.equal(torch.bincount((x >> 12) + (1 << 15)), torch.bincount((out >> 12) + (1 << 15)))
        return
    for lo in range(0, n, 1 << 28):
        s = slice(lo, min(n, lo + (1 << 28)))
        assert torch.equal(x[vo[s].long()], out[s])
    assert bool(((out[1:] > out[:-1]) | (vo[1:] > vo[:-1])).all())
    del vo
