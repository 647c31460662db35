"""CPU model of how a digit pass ranks the keys of a partial tile (csrc/radix.cu,
DigitTile::rank): half-warps take chunks of 16 x IPT keys, 16 at a time, and rank
a chunk whose sorted digits agree with one atomic per key.  The order in which
the lanes of one atomic are served is not specified, so the model serves them
from either end: whatever the order, the staged keys below `count` have to be
the tile's keys and none of its padding.  Which chunks may be ranked so is the
library's own rule (nsort_testing_unmixed_chunk)."""
import numpy as np
import pytest

import __graft_entry__
from paper_2409_03970_gb300 import nsort

HALF_WARPS = 32
PAD = 0xFFFFFFFF


@pytest.fixture(scope="module", autouse=True)
def built():
    __graft_entry__.build()


def stage(keys, count, ipt, shift, descending):
    """The tile's keys in the order of one pass, all chunks whose sorted digits
    agree and that the rule allows ranked with lanes served in the given order."""
    low = (1 << shift) - 1
    digit = (keys >> shift) & 0xFF
    chunk = 16 * ipt
    staged = np.zeros_like(keys)
    at = np.concatenate([[0], np.cumsum(np.bincount(digit, minlength=256))[:-1]])
    for c in range(HALF_WARPS):
        first = c * chunk
        free = ((keys[first] ^ keys[first + chunk - 1]) & low) == 0 and \
            nsort.nsort_testing_unmixed_chunk(first, chunk, count)
        for i in range(ipt):
            lanes = range(15, -1, -1) if free and descending else range(16)
            for lane in lanes:
                e = first + 16 * i + lane
                staged[at[digit[e]]] = keys[e]
                at[digit[e]] += 1
    return staged


@pytest.mark.parametrize("descending", [False, True])
@pytest.mark.parametrize("ipt", [4, 8, 20])
def test_no_key_lost_to_padding(ipt, descending):
    tile = HALF_WARPS * 16 * ipt
    rng = np.random.default_rng(ipt)
    for extra in range(1, 16):
        count = int(rng.integers(0, tile // 16)) * 16 + extra
        for fill in (0x7FFFFFFF, 0x00FFFFFF, None):   # i32 -1 and f32 -0.0 mapped; a high digit
            keys = np.full(tile, PAD, np.uint32)
            keys[:count] = rng.integers(0, 1 << 32, count) if fill is None else fill
            x = keys
            for shift in (0, 8, 16, 24):
                x = stage(x, count, ipt, shift, descending)
                np.testing.assert_array_equal(np.sort(x[:count]), np.sort(keys[:count]))
                x[count:] = PAD
            np.testing.assert_array_equal(x[:count], np.sort(keys[:count]))


def test_rule():
    assert nsort.nsort_testing_unmixed_chunk(64, 64, 128)       # ends with the keys
    assert nsort.nsort_testing_unmixed_chunk(128, 64, 128)      # begins behind them
    assert not nsort.nsort_testing_unmixed_chunk(64, 64, 127)
    assert not nsort.nsort_testing_unmixed_chunk(64, 64, 65)
