"""Which way plain sorts of 32-bit keys take around the end of the one-cluster
range: a cluster up to 2^16 keys, and up to 2^17 where the tile counts of the
passes don't fit in the scratch; passes else.  (Results at these sizes are in
test_gpu_digit.py.)"""
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

CLUSTER, PASSES = {"radix_cluster"}, {"radix_histogram", "radix_pass"}
# the passes' counts: 4352 bytes, and 512 for each 16,384 keys
KEYS = [(65536, CLUSTER), (65537, CLUSTER), (114_623, CLUSTER), (114_624, PASSES),
        (114_688, PASSES), (114_689, CLUSTER), (122_815, CLUSTER), (122_816, PASSES),
        (131_072, PASSES), (131_073, PASSES)]
PAIRS = [(65537, CLUSTER), (114_623, CLUSTER), (114_624, PASSES), (114_688, PASSES),
         (114_689, CLUSTER), (118_719, CLUSTER), (118_720, PASSES), (131_072, PASSES),
         (131_073, PASSES)]


@pytest.fixture(scope="module")
def ns():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2409_03970_gb300 import build, nsort
    build.build()
    nsort.lib()
    return nsort


@pytest.mark.parametrize("op,cases", [("keys", KEYS), ("pairs", PAIRS), ("pairs64", PAIRS)])
def test_routes(ns, op, cases):
    kind = {"keys": ns.KIND_KEYS, "pairs": ns.KIND_PAIRS, "pairs64": ns.KIND_PAIRS64}[op]
    for n, want in cases:
        k = torch.randint(-2**31, 2**31 - 1, (n,), dtype=torch.int32, device="cuda")
        v = torch.arange(n, dtype=torch.int64 if op == "pairs64" else torch.int32, device="cuda")
        ko, vo, tmp = torch.empty_like(k), torch.empty_like(v), ns.scratch(kind, n)
        ns.nsort_trace_enable(True)
        if op == "keys":
            rc = ns.nsort_keys(k, ko, n, ns.I32, tmp, tmp.numel())
        else:
            call = ns.nsort_pairs if op == "pairs" else ns.nsort_pairs64
            rc = call(k, v, ko, vo, n, ns.I32, tmp, tmp.numel())
        assert rc == ns.OK and ns.nsort_device_status(tmp) == ns.OK
        trace = ns.nsort_trace_read()
        ns.nsort_trace_enable(False)
        assert {t for t in trace if t.startswith(("radix", "merge"))} == want, n
        assert torch.equal(ko, k.sort()[0])
