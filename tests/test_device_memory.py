"""Device memory of the contexts, on a CUDA runtime made for tests: what is kept from one context to the next, and what
happens when the device cannot be waited for or memory runs out."""
import pytest

from fake_cuda import GLOBAL_MODE, RELAXED, FakeLibrary

TINY = dict(n_heads=4, head_dim=64, grid_h=8, grid_w=8, n_blocks=4)


@pytest.fixture
def fake():
    return FakeLibrary()


@pytest.mark.parametrize("device", [0, 63, 64, 200])
def test_every_device_index_takes_contexts(fake, device):
    fake.lib.cudaSetDevice(device)
    ctx = fake.context(**TINY)
    assert ctx.rc == 0 and ctx.append(2) == 0 and ctx.full_attend() == 0 and ctx.destroy() == 0


@pytest.mark.parametrize("mode", [0, RELAXED, GLOBAL_MODE])
def test_memory_of_a_context_destroyed_with_work_in_flight_is_not_handed_out_before_the_device_is_done(fake, mode):
    first = fake.context(**TINY)
    assert first.rc == 0 and first.append(2) == 0 and first.full_attend() == 0
    fake.work_in_flight()
    fake.capture(mode, None)  # a stream of somebody else: with it the runtime refuses to wait for the device
    assert first.destroy() == 0
    assert mode != GLOBAL_MODE or fake.busy() > 0
    fake.capture(0, None)
    second = fake.context(**TINY)
    assert second.rc == 0 and second.append(2) == 0 and second.full_attend() == 0
    assert fake.busy_writes() == 0
    assert second.destroy() == 0


def test_memory_that_could_not_be_freed_is_freed_once_the_device_can_be_waited_for(fake):
    first = fake.context(**TINY)
    assert first.append(2) == 0 and first.full_attend() == 0
    whole = fake.used()
    fake.work_in_flight()
    fake.capture(GLOBAL_MODE, None)
    assert first.destroy() == 0
    assert fake.used() == whole  # nothing could be given back
    fake.capture(0, None)
    for _ in range(3):
        again = fake.context(**TINY)
        assert again.append(2) == 0 and again.full_attend() == 0 and again.destroy() == 0
    assert fake.used() - fake.pool_unused() <= whole  # (the pool gives back by itself what exceeds its bound)
