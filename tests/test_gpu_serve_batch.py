"""GPU tests of the sort server's batches: co-batches whose requests begin and
end around the chunks of the copy kernel (1,024 keys), from many requests in a
chunk to many chunks in a request, and requests alone in their batch, whose
buffers overlap or not (the plain call, or packed), against the oracle."""
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


def request(n, pairs, seed):
    """Few distinct keys in pairs, so that stability shows."""
    k = inputs.keys(n, "u32", "uniform", seed=seed)
    return (k % 7 if pairs else k), (np.arange(n, dtype=np.uint32) if pairs else None)


def check(k, v, ko, vo):
    if v is None:
        np.testing.assert_array_equal(ko, oracle.sort_keys(k, "u32"))
        return
    wk, wv = oracle.sort_pairs(k, v, "u32")
    np.testing.assert_array_equal(ko, wk)
    np.testing.assert_array_equal(vo, wv)


def dev(x):
    return None if x is None else torch.from_numpy(x.view(np.int32)).cuda()


def host(x):
    return None if x is None else x.cpu().numpy().view(np.uint32)


@pytest.mark.parametrize("pairs", [False, True])
@pytest.mark.parametrize("sizes", [
    [1, 1], [1023, 1, 1024], [1024, 1024, 1025], [1] * 3000 + [5000] + [2] * 700,
    [65536, 3, 65535, 1021], [4096] * 9 + [1]])
def test_co_batch(ns, sizes, pairs):
    head = dev(inputs.keys(1 << 24, "u32", "uniform", seed=9))
    out = torch.empty_like(head)
    reqs = [request(n, pairs, i + 1) for i, n in enumerate(sizes)]
    bufs = [(dev(k), dev(v)) for k, v in reqs]
    outs = [(torch.empty_like(k), None if v is None else torch.empty_like(v)) for k, v in bufs]
    torch.cuda.synchronize()
    with ns.SortServer(0, 1 << 30, 1, 1 << 16) as srv:   # one stream: the rest wait behind this
        tickets = [srv.submit(head, out, dtype=0)]
        tickets += [srv.submit(k, ko, v, vo, dtype=0) for (k, v), (ko, vo) in zip(bufs, outs)]
        for t in tickets:
            assert srv.wait(t) == ns.OK
        assert all(srv.poll(t)[1]["batched"] for t in tickets[1:])
    for (k, v), (ko, vo) in zip(reqs, outs):
        check(k, v, host(ko), host(vo))


@pytest.mark.parametrize("pairs", [False, True])
@pytest.mark.parametrize("n", [1, 1025, 20001, 65536])
def test_alone(ns, n, pairs):
    k, v = request(n, pairs, n)
    with ns.SortServer(0, 1 << 28, 2, 1 << 16) as srv:
        for shift in (None, 0, n // 2):   # outputs of their own, in place, half way into the inputs
            kb, vb = (torch.zeros(2 * n, dtype=torch.int32, device="cuda") for _ in range(2))
            kb[:n] = dev(k)
            if pairs:
                vb[:n] = dev(v)
            ko, vo = ((torch.empty_like(kb[:n]), torch.empty_like(vb[:n])) if shift is None else
                      (kb[shift:shift + n], vb[shift:shift + n]))
            torch.cuda.synchronize()
            t = srv.submit(kb[:n], ko, vb[:n] if pairs else None, vo if pairs else None, dtype=0)
            assert srv.wait(t) == ns.OK and srv.poll(t)[1]["batched"]
            check(k, v, host(ko), host(vo) if pairs else None)
