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
