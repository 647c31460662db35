"""What the sort server's timing says about how a small request was sorted:
requests admitted together share t_admit and one segmented launch; one that
finds no other to join is sorted by the plain call.  Both are `batched`."""
import numpy as np
import pytest

import oracle
from paper_2409_03970_gb300 import inputs

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ns():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2409_03970_gb300 import build, nsort
    build.build()
    nsort.lib()
    return nsort


def serve(ns, reqs, head_keys):
    """Timings of the requests (arrays of u32 keys), submitted while a sort of
    head_keys keys holds the only stream, and the launches of the traced run."""
    head = torch.zeros(head_keys, dtype=torch.int32, device="cuda")
    head_out = torch.empty_like(head)
    bufs = [torch.from_numpy(k.view(np.int32)).cuda() for k in reqs]
    outs = [torch.empty_like(b) for b in bufs]
    torch.cuda.synchronize()
    with ns.SortServer(0, 4 << 30, 1, 1 << 16) as srv:
        ns.nsort_trace_enable(True)
        first = srv.submit(head, head_out, dtype=0)
        tickets = [srv.submit(b, o, dtype=0) for b, o in zip(bufs, outs)]
        for t in [first] + tickets:
            assert srv.wait(t) == ns.OK
        torch.cuda.synchronize()
        launches = {k: v["launches"] for k, v in ns.nsort_trace_read().items()}
        ns.nsort_trace_enable(False)
        timings = [srv.poll(t)[1] for t in tickets]
    for k, o in zip(reqs, outs):
        np.testing.assert_array_equal(o.cpu().numpy().view(np.uint32), oracle.sort_keys(k, "u32"))
    return timings, launches


def test_requests_that_wait_share_a_launch(ns):
    """24 requests wait behind 2^29 keys (5.6 ms; they take some 0.3 to submit)."""
    reqs = [inputs.keys(1000 + 997 * i, "u32", "uniform", seed=i) for i in range(24)]
    timings, launches = serve(ns, reqs, 1 << 29)
    assert all(t["batched"] for t in timings)
    assert len({t["t_admit"] for t in timings}) == 1
    assert launches["segmented_sort"] == 1 and "radix_cluster" not in launches


def test_a_request_alone_takes_the_plain_call(ns):
    timings, launches = serve(ns, [inputs.keys(40_000, "u32", "uniform", seed=1)], 1 << 29)
    assert timings[0]["batched"]
    assert "segmented_sort" not in launches and launches["radix_cluster"] == 1
