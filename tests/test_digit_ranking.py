"""CPU model of how a digit pass ranks the keys of a partial tile (csrc/radix.cu,
DigitTile::rank): half-warps take chunks of 16 x IPT keys, 16 at a time, and rank
a chunk whose sorted digits agree with one atomic per key.  The order in which
the lanes of one atomic are served is not specified, so the model serves them
from either end: whatever the order, the staged keys below `count` have to be
the tile's keys and none of its padding.  Who takes part in those atomics is
read from the source."""
import os
import re

import numpy as np
import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
HALF_WARPS = 32
PAD = 0xFFFFFFFF


def padding_takes_part():
    """Whether a free-order atomic of a partial tile is done for padding too."""
    with open(os.path.join(ROOT, "paper_2409_03970_gb300", "csrc", "radix.cu")) as f:
        text = re.sub(r"//[^\n]*|#pragma[^\n]*", "", f.read())
    branch = re.search(r"__all_sync\(0xffffffffu, f == l\)\) \{(.*?)\n      \} else \{", text,
                       re.S).group(1)
    full, _, partial = branch.partition("} else {")
    return not (re.match(r"\s*if \(!FREE_PARTIAL \|\| count == TILE\) \{", full) and
                "(FREE_PARTIAL || count == TILE) && __all_sync" in text and
                re.search(r"if \(e0 \+ 16 \* i < count\)\s*stage\[", partial))


def stage(keys, count, ipt, shift, descending):
    """The tile's keys in the order of one pass, every chunk whose sorted digits
    agree ranked with the lanes served in the given order; PAD where nothing
    is staged."""
    low = (1 << shift) - 1
    digit = (keys >> shift) & 0xFF
    chunk = 16 * ipt
    staged = np.full_like(keys, PAD)
    counts = np.stack([np.bincount(digit[c * chunk:(c + 1) * chunk], minlength=256)
                       for c in range(HALF_WARPS)])
    start = np.concatenate([[0], np.cumsum(counts.sum(0))[:-1]])   # the digit's place in the tile
    pads = padding_takes_part()
    for c in range(HALF_WARPS):
        at = start + counts[:c].sum(0)                             # this half-warp's counters
        first = c * chunk
        free = ((keys[first] ^ keys[first + chunk - 1]) & low) == 0
        for i in range(ipt):
            for lane in range(15, -1, -1) if free and descending else range(16):
                e = first + 16 * i + lane
                if free and not pads and e >= count:
                    continue
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
