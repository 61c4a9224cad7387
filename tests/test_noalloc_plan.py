"""How the allocation-free call spreads query-tile pairs over the SMs (host code, on a CUDA runtime made for tests)."""
import ctypes as C
import random

import pytest

from fake_cuda import FakeLibrary
from test_gpu_noalloc_cuts import CASES


@pytest.mark.parametrize("pairs,tiles,line_at_64,line_at_128", [
    (130, 200, True, False), (130, 120, True, False), (120, 120, True, False), (80, 16, True, False), (90, 20, True, False),
    (400, 80, True, False),                                                             # slower as a line at head_dim 128
    (75, 24, True, True), (100, 56, True, True), (110, 120, True, True), (200, 40, True, True), (450, 56, True, True),  # faster at both
    (140, 56, False, False), (296, 80, False, False), (148, 200, False, False)])       # waves that are full
def test_pairs_are_laid_on_a_line_where_that_was_measured_to_be_faster(pairs, tiles, line_at_64, line_at_128):
    fake = FakeLibrary()
    assert (fake.noalloc_cuts(pairs, 128 * tiles, 148, 64) == -1) == line_at_64
    assert (fake.noalloc_cuts(pairs, 128 * tiles, 148, 128) == -1) == line_at_128


@pytest.mark.parametrize("heads,n_q,tiles,pieces", CASES)
def test_the_cases_that_run_on_the_gpu_are_cut_as_they_say(heads, n_q, tiles, pieces):
    fake = FakeLibrary()
    for head_dim in (64, 128):
        for n_keys in (128 * tiles, 128 * tiles - 127):
            assert fake.noalloc_cuts(heads * -(-n_q // 256), n_keys, 148, head_dim) == pieces


def test_shares_of_every_plan_fit_the_fixed_scratch():
    """Any number of pairs, key tiles and SMs: shares in order, none empty, all of the line; a CTA leaves at most two partial results,
    all CTAs no more than there are slots; a pair's pieces are no shorter than four tiles on a line; entries to merge fit."""
    fake, rng = FakeLibrary(), random.Random(1)
    begins, slots, entries, cut = (C.c_longlong * 1025)(), C.c_int(), C.c_int(), {0: 0, 1: 0, -1: 0}
    for trial in range(4000):
        pairs = int(round(2048 ** rng.random())) if trial % 2 else rng.randint(30, 600)
        tiles, n_sm, head_dim = int(round(700 ** rng.random())), rng.choice([148, 148, 148, 132, 74, 16, 160, 1024]), rng.choice([64, 128])
        n = fake.noalloc_shares(pairs, 128 * tiles - rng.randint(0, 127), n_sm, head_dim, begins, C.byref(slots), C.byref(entries))
        kind = fake.noalloc_cuts(pairs, 128 * tiles, n_sm, head_dim)
        cut[min(kind, 1)] += 1
        if kind == 0:
            assert n == 0
            continue
        b = begins[: n + 1]
        assert n <= min(n_sm, 148) and b[0] == 0 and b[n] == pairs * tiles and all(x < y for x, y in zip(b, b[1:]))
        partial = merged = 0
        for x, y in zip(b, b[1:]):
            pieces = [(max(x, p * tiles), min(y, (p + 1) * tiles)) for p in range(x // tiles, (y - 1) // tiles + 1)]
            short = [e - s for s, e in pieces if e - s < tiles]
            assert len(short) <= 2 and (kind > 0 or all(t >= 4 for t in short))
            partial += len(short)
            merged += sum(s % tiles == 0 and e - s < tiles for s, e in pieces)
        assert partial <= slots.value and 2 * merged <= entries.value
        if kind > 0:
            assert n == pairs * kind and merged == pairs
    assert min(cut.values()) > 300
