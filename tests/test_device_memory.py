"""Device memory of the contexts, on a CUDA runtime made for tests: what is kept from one context to the next, and what
happens when the device cannot be waited for or memory runs out."""
import os
import re

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


@pytest.mark.parametrize("idle_blocks,heads", [(False, 5), (False, 16), (True, 5), (True, 16)])
def test_creation_takes_back_all_that_the_library_keeps_idle(fake, idle_blocks, heads):
    wanted = dict(TINY, n_heads=heads)  # 5: memory runs out at its monolithic cache, 16: later, at its blocks
    clean = FakeLibrary()
    need = clean.context(**wanted) and clean.used()
    contexts = [fake.context(**TINY) for _ in range(3)]
    for ctx in contexts:
        if idle_blocks:  # blocks, scratch arrays among them, and the monolithic cache in the pool
            assert ctx.append(2) == 0 and ctx.full_attend() == 0 and ctx.destroy() == 0
        else:  # the monolithic cache only, the blocks are in use
            assert ctx.append() == 0 and ctx.split([0, 1, 2, 3]) == 0
    idle = fake.used() if idle_blocks else fake.pool_unused()
    assert idle > fake.pool_unused() > 0 if idle_blocks else idle > 0
    fake.capacity_left(need - idle)  # every idle byte has to come back for this one to fit
    assert fake.context(**wanted).rc == 0


def test_a_growing_scratch_array_takes_back_the_pools_idle_memory(fake):
    ctx = fake.context(**TINY)
    gone = fake.context(**TINY)
    assert ctx.append(2) == 0 and gone.append() == 0 and gone.split([0, 1, 2, 3]) == 0
    assert fake.pool_unused() > 0
    clean = FakeLibrary()
    twin = clean.context(**TINY)
    twin.append(2)
    before = clean.used()
    assert twin.full_attend() == 0
    fake.capacity_left(max(0, clean.used() - before - fake.pool_unused()))
    assert ctx.full_attend() == 0


def test_scratch_may_grow_beside_the_capture_of_another_stream(fake):
    ctx = fake.context(n_heads=6, head_dim=128, grid_h=13, grid_w=22, n_blocks=4)
    assert ctx.append(1) == 0 and ctx.full_attend(stream=78) == 0
    first = fake.attn_part_o()
    assert fake.is_live(first)
    fake.capture(RELAXED, 77)
    assert ctx.append(3) == 0 and ctx.full_attend(stream=78) == 0
    assert fake.attn_part_o() != first and fake.is_live(fake.attn_part_o())
    assert not fake.capture_invalidated()
    fake.capture(0, None)
    twin = fake.context(n_heads=6, head_dim=128, grid_h=13, grid_w=22, n_blocks=4)
    assert twin.append(1) == 0 and twin.full_attend() == 0 and fake.attn_part_o() == first  # it was kept for others


@pytest.mark.parametrize("refusal", ["memory", "capture"])
def test_a_list_that_is_already_uploaded_has_its_scratch_after_anothers_growth_failed(fake, refusal):
    ctx = fake.context(n_heads=6, head_dim=128, grid_h=13, grid_w=22, n_blocks=4, cell_h=6, cell_w=6, keep_monolithic=1)
    assert ctx.append(4) == 0 and ctx.split([0, 1, 2, 3, 2, 3]) == 0 and ctx.attend() == 0
    first = fake.attn_part_o()
    if refusal == "memory":
        fake.capacity_left(64 << 10)  # enough for the dense list, not for its partial results
        assert ctx.full_attend() == -4
    else:
        fake.capture(GLOBAL_MODE, 77)
        assert ctx.full_attend(stream=78) != 0
        fake.capture(0, None)
    assert ctx.attend() == 0
    assert fake.is_live(fake.attn_part_o())
    assert refusal == "memory" or fake.attn_part_o() == first


def test_nothing_kept_from_before_a_device_reset_comes_back(fake):
    for _ in range(2):
        old = fake.context(**TINY)
        assert old.append(2) == 0 and old.full_attend() == 0 and old.destroy() == 0
        fake.device_reset()
        new = fake.context(**TINY)
        assert new.rc == 0 and new.append(2) == 0 and new.full_attend() == 0
        assert fake.stray_writes() == 0
        assert new.destroy() == 0


def test_kept_memory_can_be_given_back(fake):
    alive = fake.context(**TINY)
    with_one = fake.used()
    gone = [fake.context(**TINY) for _ in range(3)]
    for ctx in gone:
        assert ctx.append(2) == 0 and ctx.full_attend() == 0 and ctx.destroy() == 0
    assert fake.used() > with_one
    assert fake.lib.headcast_release_memory() == 0 and fake.used() == with_one
    assert alive.append(2) == 0 and alive.full_attend() == 0 and alive.destroy() == 0
    fake.capture(RELAXED, None)
    assert fake.lib.headcast_release_memory() == -3
    fake.capture(0, None)
    assert fake.lib.headcast_release_memory() == 0 and fake.used() == 0


def test_the_header_states_what_is_kept():
    root = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
    source = open(os.path.join(root, "paper_2607_20125_b200", "csrc", "context.h")).read()
    kept = [int(re.search(name + r" = (?:size_t\()?(\d+)(?:\)|ull) << 20;", source).group(1)) for name in ("CACHE_KEEP_BYTES", "MONO_KEEP_BYTES")]
    assert f"at most {sum(kept)} MB per GPU" in open(os.path.join(root, "include", "headcast.h")).read()


def test_scratch_that_a_graph_uses_stays_when_another_list_needs_more(fake):
    ctx = fake.context(n_heads=6, head_dim=128, grid_h=13, grid_w=22, n_blocks=4, cell_h=6, cell_w=6, keep_monolithic=1)
    assert ctx.append(4) == 0 and ctx.split([0, 1, 2, 3, 2, 3]) == 0 and ctx.attend() == 0
    fake.capture(RELAXED, 21)
    assert ctx.attend(stream=21) == 0
    fake.capture(0, None)
    in_graph = fake.attn_part_o()
    fake.capacity_left(64 << 10)
    assert ctx.full_attend() == -4 and fake.is_live(in_graph)  # not even for want of memory
    fake.capacity_left(64 << 20)
    assert ctx.full_attend() == 0 and fake.attn_part_o() != in_graph and fake.is_live(in_graph)
    assert ctx.destroy() == 0 and fake.lib.headcast_release_memory() == 0 and fake.used() == 0


def test_the_allocation_free_call_finds_its_array_again_after_a_device_reset(fake):
    import ctypes
    buffer = ctypes.create_string_buffer(64)
    x = (ctypes.addressof(buffer) + 15) & ~15
    for _ in range(3):
        for _ in range(2):
            assert fake.lib.headcast_dense_attend_noalloc(x, x, x, x, 100, 100, 4, 64, 0.0, None) == 0
            assert fake.noalloc_list_is_the_devices()
        fake.device_reset()
