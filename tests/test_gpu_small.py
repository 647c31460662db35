"""One-tile sorts (csrc/small.cu) against the oracle, bit for bit: every size
at which the shape of the CTA changes and at the edges of a warp's share of
each shape, all types, in place and on buffers of any alignment, with keys
equal to the padding.  Sorts are exact: no tolerance."""
import numpy as np
import pytest

import oracle
from paper_2409_03970_gb300 import inputs

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

CODE = {"u32": 0, "i32": 1, "f32": 2, "u64": 3, "i64": 4, "f64": 5}
SIZES = [1, 2, 31, 32, 33, 255, 256, 257, 511, 512, 513, 767, 768, 769, 1023, 1024, 1025, 1280, 1281,
         1792, 1793, 2047, 2048, 2049, 3072, 3073, 4095, 4096, 4097, 5120, 6145, 7169, 8191, 8192,
         8193, 9216, 12289, 16383, 16384]


@pytest.fixture(scope="module")
def ns():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2409_03970_gb300 import build, nsort
    build.build()
    nsort.lib()
    return nsort


def cuda(a, offset):
    t = {4: torch.int32, 8: torch.int64}[a.dtype.itemsize]
    x = torch.full((a.size + offset + 8,), 0x5A5A5A5A, dtype=t, device="cuda")
    x[offset:offset + a.size] = torch.from_numpy(a.view({4: np.int32, 8: np.int64}[a.dtype.itemsize]))
    return x[offset:]


def host(t, n, like):
    assert bool((t[n:] == 0x5A5A5A5A).all()), "wrote past the output"
    return t[:n].cpu().numpy().view(like.dtype)


def ones_at(x, seed):
    """Some keys equal to the padding (the largest key)."""
    x = x.copy()
    x[inputs.counter_u32(seed, 2, 0, x.size) % 7 == 0] = np.iinfo(x.dtype).max
    return x


@pytest.mark.parametrize("dt", list(CODE))
def test_keys(ns, dt):
    wide = dt in inputs.KEY64_DTYPES
    for n in SIZES:
        if wide and n > 4096:
            continue
        for i, dist in enumerate(["uniform", "dup16", "reverse"]):
            x = inputs.keys64(n, dt, dist, n) if wide else inputs.keys(n, dt, dist, n)
            if i == 1:
                x = ones_at(x, n)
            want = oracle.sort_keys64(x, dt) if wide else oracle.sort_keys(x, dt)
            k = cuda(x, (n + i) % 4)
            ko = k if i == 2 else cuda(np.zeros_like(x), n % 4)
            assert ns.nsort_keys(k, ko, n, CODE[dt], None, 0) == ns.OK
            np.testing.assert_array_equal(host(ko, n, x), want, err_msg=f"{n} {dist}")


@pytest.mark.parametrize("dt", ["u32", "i32", "f32"])
@pytest.mark.parametrize("vbytes", [4, 8])
def test_pairs(ns, dt, vbytes):
    for n in SIZES:
        if n > 8192:
            continue
        for i, dist in enumerate(["uniform", "dup16", "reverse"]):
            x = inputs.keys(n, dt, dist, n)
            if i == 1:
                x = ones_at(x, n)
            order = np.arange(n, dtype=np.uint32)
            wk, perm = oracle.sort_pairs(x, order, dt)
            v = order if vbytes == 4 else inputs.counter_u64(n, 7, 0, n)
            off = (n + i) % 4 if vbytes == 4 else 0   # (pairs64: aligned outputs only)
            k, vt = cuda(x, off), cuda(v, off)
            ko = k if i == 2 else cuda(np.zeros_like(x), off)
            vo = vt if i == 2 else cuda(np.zeros_like(v), off)
            call = ns.nsort_pairs if vbytes == 4 else ns.nsort_pairs64
            assert call(k, vt, ko, vo, n, CODE[dt], None, 0) == ns.OK
            np.testing.assert_array_equal(host(ko, n, x), wk, err_msg=f"{n} {dist}")
            np.testing.assert_array_equal(host(vo, n, v), v[perm], err_msg=f"{n} {dist}")
