"""Failure detection in the digit passes without a GPU fault: their waits for
other tiles' counts give up after a limit, the status word says so, no key of
the tile is written and the context keeps working."""
import time

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


def run(ns, which, limit_us):
    """(first tile's status, second tile's, whether the destination is untouched, seconds)"""
    tmp = torch.zeros(ns.SELFTEST_DIGIT_BYTES, dtype=torch.uint8, device="cuda")
    torch.cuda.synchronize()
    t0 = time.perf_counter()
    assert ns.nsort_selftest_digit_waits(which, tmp, limit_us) == ns.OK
    torch.cuda.synchronize()
    seconds = time.perf_counter() - t0
    host = tmp.cpu().numpy()
    keys = 3 * 512 * {0: 32, 1: 20, 2: 4 * 8}[which]
    first, second = host[:16].view(np.int32)[[0, 2]]
    return first, second, bool((host[256:256 + 4 * keys] == 0xA5).all()), seconds


@pytest.mark.parametrize("which", [0, 1, 2])
def test_waits_give_up_and_report(ns, which):
    run(ns, which, 1000)                             # (kernels loaded)
    first, _, _, seconds = run(ns, which, 20_000)
    assert first == ns.ETIMEOUT
    assert 0.02 <= seconds < 5.0
    n = 6_000_011
    x = inputs.keys(n, "f32", "uniform", seed=31)
    xt = torch.from_numpy(x.view(np.int32)).cuda()
    out = torch.empty_like(xt)
    sc = ns.scratch(ns.KIND_KEYS, n)
    assert ns.nsort_keys(xt, out, n, ns.F32, sc, sc.numel()) == ns.OK
    assert ns.nsort_device_status(sc) == ns.OK
    np.testing.assert_array_equal(out.cpu().numpy().view(np.uint32), oracle.sort_keys(x, "f32"))


@pytest.mark.parametrize("which", [0, 1, 2])
def test_later_tiles_do_not_build_on_a_wait_that_gave_up(ns, which):
    """The tile after the one that gave up (its launch begins when that has
    ended) gives up as well, and neither writes a key."""
    first, second, untouched, seconds = run(ns, which, 20_000)
    assert (first, second) == (ns.ETIMEOUT, ns.ETIMEOUT)
    assert untouched and seconds < 5.0
