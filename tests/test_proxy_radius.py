"""Host-only: the radius that the Spatial proxy's kernel is given never exceeds what reaches the whole frame, so its loop over
grid rows ends and its products fit 32 bits whatever the configuration asks for."""
import pytest

from fake_cuda import FakeLibrary


@pytest.mark.parametrize("gh,gw", [(16, 17), (8, 8), (1, 300), (300, 1)])
@pytest.mark.parametrize("radius", [0, 2, 299, 300, 400, 2**31 - 1])
def test_radius_of_the_proxy_launch(gh, gw, radius):
    fake = FakeLibrary()
    ctx = fake.context(n_heads=4, head_dim=64, grid_h=gh, grid_w=gw, n_blocks=3, proxy_radius=radius)
    assert ctx.rc == 0 and ctx.append(2) == 0 and ctx.classify() == 0
    assert fake.attn_radius() == min(radius, max(gh, gw))
