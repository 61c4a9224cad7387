"""An error of the CUDA runtime is reported by the call that met it, or dealt with there; no later call reports it again.  On a
CUDA runtime made for tests."""
import pytest

from fake_cuda import GLOBAL_MODE, RELAXED, FakeLibrary

TINY = dict(n_heads=4, head_dim=64, grid_h=8, grid_w=8, n_blocks=4, keep_monolithic=1)


@pytest.mark.parametrize("how", ["capture", "memory", "destroy beside a capture", "growth beside a capture", "release beside a capture", "create"])
def test_a_refusal_shows_up_once(how):
    fake = FakeLibrary()
    ctx, other = fake.context(**TINY), fake.context(**TINY)
    assert ctx.append(1) == 0 and ctx.export() == 0
    if how == "capture":
        fake.capture(GLOBAL_MODE, 99)
        assert ctx.full_attend() == -3
    elif how == "memory":
        fake.capacity_left(0)
        assert ctx.append(3) == 0 and ctx.full_attend() == -4
    elif how == "destroy beside a capture":
        fake.capture(RELAXED, 99)
        assert other.append(2) == 0 and other.destroy() == 0
    elif how == "growth beside a capture":
        assert ctx.full_attend() == 0 and other.append(4) == 0 and other.full_attend() == 0 and other.destroy() == 0
        assert ctx.append(3) == 0  # what its lists need lies in the memory that the other has left
        fake.capture(GLOBAL_MODE, 99)
        ctx.full_attend()
    elif how == "create":
        fake.capacity_left(0)
        assert fake.context(**dict(TINY, n_heads=8)).rc == -4
    else:
        fake.capture(RELAXED, 99)
        assert fake.lib.headcast_release_memory() == -3
    fake.capture(0, None)
    assert ctx.export() == 0
