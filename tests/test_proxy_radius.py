"""Host-only: the Spatial proxy's launch.  The radius that the kernel is given never exceeds what reaches the whole frame, so its
loop over grid rows ends and its products fit 32 bits whatever the configuration asks for; and dealing the query pairs per
frame never sweeps more key tiles than pairs of 256 across the block with bands of whole grid rows."""
import pytest

from fake_cuda import FakeLibrary


@pytest.mark.parametrize("gh,gw", [(16, 17), (8, 8), (1, 300), (300, 1)])
@pytest.mark.parametrize("radius", [0, 2, 299, 300, 400, 2**31 - 1])
def test_radius_of_the_proxy_launch(gh, gw, radius):
    fake = FakeLibrary()
    ctx = fake.context(n_heads=4, head_dim=64, grid_h=gh, grid_w=gw, n_blocks=3, proxy_radius=radius)
    assert ctx.rc == 0 and ctx.append(2) == 0 and ctx.classify() == 0
    assert fake.attn_radius() == min(radius, max(gh, gw))


def tile_steps_of_whole_rows(gh, gw, radius, frames, heads, filled):
    t_f, steps = gh * gw, 0
    for q0 in range(0, frames * t_f, 256):
        q1 = min(frames * t_f, q0 + 256) - 1
        keys = t_f
        if q0 // t_f == q1 // t_f:
            keys = (min(gh - 1, q1 % t_f // gw + radius) + 1 - max(0, q0 % t_f // gw - radius)) * gw
        steps += -(-keys // 128)
    return steps * frames * filled * heads


@pytest.mark.parametrize("gh,gw", [(1, 300), (300, 1), (16, 16), (17, 16), (16, 17), (1, 257), (20, 15), (19, 27), (27, 19), (30, 52), (2, 200)])
@pytest.mark.parametrize("radius", [0, 2, 9, 400])
def test_no_deal_of_the_query_pairs_sweeps_more(gh, gw, radius):
    fake = FakeLibrary()
    ctx = fake.context(n_heads=2, head_dim=64, grid_h=gh, grid_w=gw, n_blocks=3, proxy_radius=radius)
    assert ctx.append(2) == 0 and ctx.classify() == 0
    assert fake.attn_tile_steps() <= tile_steps_of_whole_rows(gh, gw, radius, 3, 2, 2)
