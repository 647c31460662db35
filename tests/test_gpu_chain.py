"""GPU tests of small sorts that follow one another on a stream, each reading
what the one before it writes: their kernels are launched before their
predecessors end and wait for them, alone and captured in a CUDA graph, among
kernels of other libraries."""
import numpy as np
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


@pytest.mark.parametrize("captured", [False, True])
@pytest.mark.parametrize("n", [33, 1000, 8192, 16384, 60000, 200003])
def test_chain(ns, n, captured):
    """x -> sorted by rank of a permutation -> its payloads sorted back: the
    chain gives the permutation's inverse, then the identity, whatever was in
    the buffers before."""
    s, side = torch.cuda.Stream(), torch.cuda.Stream()
    perm, k1, v1, k2, v2, back = (torch.empty(n, dtype=torch.int32, device="cuda")
                                  for _ in range(6))
    ident = torch.arange(n, dtype=torch.int32, device="cuda")
    tp, tk = ns.scratch(ns.KIND_PAIRS, n), ns.scratch(ns.KIND_KEYS, n)
    out = torch.empty(4, n, dtype=torch.int32, device="cuda")

    def chain():
        for r in range(4):
            assert ns.nsort_pairs(perm, ident, k1, v1, n, ns.U32, tp, tp.numel(), s) == ns.OK
            assert ns.nsort_pairs(v1, k1, k2, v2, n, ns.U32, tp, tp.numel(), s) == ns.OK
            assert ns.nsort_keys(v2, back, n, ns.U32, tk, tk.numel(), s) == ns.OK
            out[r].copy_(v2)
            side.wait_stream(s)
            with torch.cuda.stream(side):
                out[r] += back
            s.wait_stream(side)
            perm.copy_((v2 + 1) % n)        # the next round's permutation

    first = np.random.RandomState(n).permutation(n).astype(np.int32)
    torch.cuda.synchronize()
    with torch.cuda.stream(s):
        perm.copy_(torch.from_numpy(first))
        chain()
        s.synchronize()
        if captured:
            for b in (k1, v1, k2, v2, back):
                b.fill_(-1)
            g = torch.cuda.CUDAGraph()
            with torch.cuda.graph(g, stream=s):
                chain()
            perm.copy_(torch.from_numpy(first))
            g.replay()
        s.synchronize()
    # sorting (perm, i) gives v1 = inverse(perm); sorting (v1, perm sorted) gives perm again
    want = first.astype(np.int64)
    for r in range(4):
        np.testing.assert_array_equal(out[r].cpu().numpy(), want + np.arange(n))
        want = (want + 1) % n
