"""Sorts on one stream beside a queue of small sorts on another: the queue's
kernels that wait for their turn must not take the SMs that the other stream's
sorts need."""
import pytest

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


def pairs(ns, n, stream):
    k, v = (torch.randint(-2**31, 2**31 - 1, (n,), dtype=torch.int32, device="cuda") for _ in "kv")
    ko, vo, tmp = torch.empty_like(k), torch.empty_like(v), ns.scratch(ns.KIND_PAIRS, n)

    def call():
        assert ns.nsort_pairs(k, v, ko, vo, n, ns.U32, tmp, tmp.numel(), stream.cuda_stream) == ns.OK
    return call


@pytest.mark.parametrize("queued", [8192, 60_000])
def test_queue_leaves_the_other_stream_its_sms(ns, queued):
    """Four sorts of 200,003 pairs take about as long beside a queue of one-tile
    or one-cluster sorts as alone.  (Beside clusters that each let the next one
    in at its start such sorts took up to 2.5 times as long.)"""
    sa, sb = torch.cuda.Stream(), torch.cuda.Stream()
    a, b = pairs(ns, queued, sa), pairs(ns, 200_003, sb)

    def once(queue):
        gate, t0, t1 = (torch.cuda.Event(enable_timing=True) for _ in range(3))
        torch.cuda.synchronize()
        with torch.cuda.stream(sa):
            torch.cuda._sleep(10_000_000)      # some milliseconds, for the queue to build up behind
            gate.record()
        for _ in range(queue):
            a()
        with torch.cuda.stream(sb):
            sb.wait_event(gate)
            torch.cuda._sleep(100_000)         # the queue is under way
            t0.record()
            for _ in range(4):
                b()
            t1.record()
        torch.cuda.synchronize()
        return t0.elapsed_time(t1)

    for q in (0, 80):
        once(q)
    alone = sorted(once(0) for _ in range(9))[4]
    beside = sorted(once(80) for _ in range(9))[4]
    assert beside < 1.6 * alone, (alone, beside)
