"""Scratch of the four-way merge passes (CPU): the boundary records of every
pass of a plan fit in what nsort_temp_bytes asks for.  A pass over runs of `run`
keys writes tpg + 1 records of 4 int64 for each group of four runs, the last
one partial or not (csrc/nsort.cu, merge4_bounds_kernel)."""
import random

import pytest

import __graft_entry__
from paper_2409_03970_gb300 import nsort

TILE, SAMPLE, SAMPLES_PER_TILE = 16384, 64, 64


def align(x):
    return -(-x // 256) * 256


def temp_bytes(n, four_way):
    prev = nsort.nsort_testing_set_four_way_min(0 if four_way else nsort.FOUR_WAY_NEVER)
    try:
        return nsort.nsort_temp_bytes(nsort.KIND_KEYS, n)
    finally:
        nsort.nsort_testing_set_four_way_min(prev)


def records(n, run):
    """Boundary records of one pass."""
    tpg = -(-4 * (run // SAMPLE) // SAMPLES_PER_TILE)
    return -(-n // (4 * run)) * (tpg + 1)


def sizes():
    rng = random.Random(1)
    yield from (2 * TILE + 1, 4 * TILE, 4 * TILE + 1, (1 << 20) + 1, (1 << 22) + 9, (1 << 26) + 1, 1 << 28)
    for _ in range(200):
        yield int(2 ** rng.uniform(15.1, 31))


@pytest.fixture(scope="module", autouse=True)
def built():
    __graft_entry__.build()


def test_boundary_records_of_every_pass_fit():
    for n in sizes():
        levels = max(0, (-(-n // TILE) - 1).bit_length())
        if levels < 2:
            continue
        run = TILE << (levels % 2)                  # a one-level pass first if they are odd
        need = 0
        while run < n:
            need = max(need, records(n, run) * 4 * 8)
            run *= 4
        # behind the two-way plan's arrays: a merged sample record of 8 bytes a sample, then these
        room = temp_bytes(n, True) - temp_bytes(n, False) - align((n // SAMPLE + 2) * 8)
        assert room >= need, n
