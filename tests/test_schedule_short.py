"""Host-only: short work lists (fewer items than SMs) are cut so that no SM walks a long key range alone, and still cover
every (head, query row, key tile) once."""
import numpy as np
import pytest

from paper_2607_20125_b200 import binding, synth
from test_schedule_host import F, check_plan


@pytest.mark.parametrize("gh,gw,heads,d,blocks,cell,longest", [
    # longest: key tiles that one SM may walk, of headcast_attend and of headcast_full_attend; uncut it would be
    (8, 8, [0, 1, 2, 3], 64, 5, 10, (1, 1)),           # 8 and 8: one query-tile pair per head
    (13, 22, [0, 1, 2, 3, 2, 3], 128, 4, 6, (3, 5)),   # 27 and 27: ragged tiles and cells
    (1, 1, [3], 64, 2, 10, (1, 1)),                    # 1 and 1: one token per frame, nothing to cut
    (9, 12, [3] * 8, 128, 4, 10, (2, 2)),              # 11 and 11
    (17, 19, [3, 3, 2, 2, 0, 1], 128, 8, 5, (6, 11)),  # 61 and 61; evenly spread 4.6 and 9.9
])
def test_no_sm_walks_a_long_key_range_alone(gh, gw, heads, d, blocks, cell, longest):
    w = synth.Workload("short", len(heads), d, gh, gw, blocks, cell_h=cell, cell_w=cell, labels=tuple(heads))
    for dense in (False, True):
        items, _ = check_plan(w, heads, blocks, 148, dense)
        _, first = binding.plan_schedule(binding.default_config(
            n_heads=len(heads), head_dim=d, grid_h=gh, grid_w=gw, n_blocks=blocks, cell_h=cell, cell_w=cell), heads, blocks, 148, dense)
        tiles = items[:, F["tile_end"]] - items[:, F["tile_begin"]]
        per_cta = np.array([tiles[first[b]:first[b + 1]].sum() for b in range(148)])
        assert per_cta.max() <= longest[dense], (dense, per_cta.max())
