"""How the allocation-free call spreads query-tile pairs over the SMs (host code, on a CUDA runtime made for tests)."""
import pytest

from fake_cuda import FakeLibrary


@pytest.mark.parametrize("pairs,tiles,line_at_64,line_at_128", [
    (130, 200, True, False), (130, 120, True, False), (120, 120, True, False), (80, 16, True, False), (90, 20, True, False),
    (400, 80, True, False),                                                             # slower as a line at head_dim 128
    (75, 24, True, True), (100, 56, True, True), (110, 120, True, True), (200, 40, True, True), (450, 56, True, True),  # faster at both
    (140, 56, False, False), (296, 80, False, False), (148, 200, False, False)])       # waves that are full
def test_pairs_are_laid_on_a_line_where_that_was_measured_to_be_faster(pairs, tiles, line_at_64, line_at_128):
    fake = FakeLibrary()
    assert (fake.noalloc_cuts(pairs, 128 * tiles, 148, 64) == -1) == line_at_64
    assert (fake.noalloc_cuts(pairs, 128 * tiles, 148, 128) == -1) == line_at_128
