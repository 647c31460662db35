"""The warp-group sorts of nsort_segmented against the oracle, bit for bit:
segments whose lengths lie at the edges of a warp's share (1024 keys, 512
pairs), of the groups of 1, 2, 4, 8 and 16 warps, and of the merge levels
above them, with few and with many items in the queue.  Sorts are exact: no
tolerance."""
import numpy as np
import pytest

import oracle
from paper_2409_03970_gb300 import inputs

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

CODE = {"u32": 0, "i32": 1, "f32": 2}
EDGES = [512, 1024, 1536, 2048, 3072, 4096, 5120, 7168, 8192, 9216, 12288, 16384, 17408, 20480,
         24576, 32768, 33792]


@pytest.fixture(scope="module")
def ns():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2409_03970_gb300 import build, nsort
    build.build()
    nsort.lib()
    cfg = nsort.nsort_segmented_get_config()
    yield nsort
    nsort.nsort_segmented_set_config(**cfg)


@pytest.mark.parametrize("threads", [256, 512])
@pytest.mark.parametrize("pairs", [False, True], ids=["keys", "pairs"])
@pytest.mark.parametrize("dt,dist,copies", [("u32", "uniform", 8), ("i32", "dup16", 1),
                                            ("f32", "sorted", 1), ("f32", "reverse", 3)])
def test_group_edges(ns, dt, dist, copies, pairs, threads):
    lens = [e + d for e in EDGES for d in (-1, 0, 1)] * copies + [0, 1, 17, 300]
    lens = np.array(lens)[np.argsort(inputs.counter_u32(3, 1, 0, len(lens)), kind="stable")]
    off = np.zeros(lens.size + 1, np.int64)
    np.cumsum(lens, out=off[1:])
    n = int(off[-1])
    keys = inputs.keys(n, dt, dist, seed=n)
    vals = np.arange(n, dtype=np.uint32)
    assert ns.nsort_segmented_set_config(block_threads=threads) == ns.OK
    k = torch.from_numpy(keys.view(np.int32)).cuda()
    v = torch.from_numpy(vals.view(np.int32)).cuda() if pairs else None
    ko, vo = torch.empty_like(k), torch.empty_like(v) if pairs else None
    o = torch.from_numpy(off).cuda()
    kind = ns.KIND_SEGMENTED_PAIRS if pairs else ns.KIND_SEGMENTED
    need = ns.nsort_temp_bytes(kind, n, lens.size)
    tmp = torch.full((need + 256,), 0x5A, dtype=torch.uint8, device="cuda")   # any contents
    rc = ns.nsort_segmented(k, ko, v, vo, o, lens.size, n, CODE[dt], tmp, need)
    assert rc == ns.OK and ns.nsort_device_status(tmp) == ns.OK
    assert bool((tmp[need:] == 0x5A).all()), "wrote past the scratch"
    got = ko.cpu().numpy().view(np.uint32)
    got_v = vo.cpu().numpy().view(np.uint32) if pairs else None
    for a, b in zip(off[:-1], off[1:]):
        if pairs:
            wk, wv = oracle.sort_pairs(keys[a:b], vals[a:b], dt)
            np.testing.assert_array_equal(got_v[a:b], wv, err_msg=f"{b - a}")
        else:
            wk = oracle.sort_keys(keys[a:b], dt)
        np.testing.assert_array_equal(got[a:b], wk, err_msg=f"{b - a}")


@pytest.mark.parametrize("pairs", [False, True], ids=["keys", "pairs"])
@pytest.mark.parametrize("nseg", [1, 255, 256, 257, 513, 1300])
def test_binning(ns, nseg, pairs):
    """Segments of every bin in each CTA of the binning and at its edges; calls
    that follow one another in one scratch, the first of malformed offsets."""
    lens = np.array([0, 1, 16, 17, 256, 257, 1024, 1025, 2048, 4096, 8192, 8193, 16385, 40000])
    lens = lens[inputs.counter_u32(nseg, 1, 0, nseg) % lens.size]
    lens[-1] = 33000
    off = np.zeros(nseg + 1, np.int64)
    np.cumsum(lens, out=off[1:])
    n = int(off[-1])
    bad = off.copy()
    bad[-1] = n - 1
    keys = inputs.keys(n, "u32", "uniform", seed=n) >> np.uint32(20)
    k = torch.from_numpy(keys.view(np.int32)).cuda()
    v = torch.arange(n, dtype=torch.int32, device="cuda") if pairs else None
    ko, vo = torch.empty_like(k), torch.empty_like(v) if pairs else None
    kind = ns.KIND_SEGMENTED_PAIRS if pairs else ns.KIND_SEGMENTED
    tmp = torch.full((ns.nsort_temp_bytes(kind, n, nseg),), 0x5A, dtype=torch.uint8, device="cuda")
    for offsets in (bad, off, off):
        o = torch.from_numpy(offsets).cuda()
        assert ns.nsort_segmented(k, ko, v, vo, o, nseg, n, 0, tmp, tmp.numel()) == ns.OK
    assert ns.nsort_device_status(tmp) == ns.OK
    got = ko.cpu().numpy().view(np.uint32)
    got_v = vo.cpu().numpy().view(np.uint32) if pairs else None
    for a, b in zip(off[:-1], off[1:]):
        if pairs:
            wk, wv = oracle.sort_pairs(keys[a:b], np.arange(a, b, dtype=np.uint32), "u32")
            np.testing.assert_array_equal(got_v[a:b], wv)
        else:
            wk = oracle.sort_keys(keys[a:b], "u32")
        np.testing.assert_array_equal(got[a:b], wk)
