"""Calls of one context on several streams, on a CUDA runtime made for tests: launches that share the context's scratch memory
follow one another, or use a scratch of their own."""
import pytest

from fake_cuda import RELAXED, FakeLibrary

SIZES = [dict(n_heads=4, head_dim=64, grid_h=8, grid_w=8, n_blocks=5, keep_monolithic=1),     # short lists
         dict(n_heads=6, head_dim=128, grid_h=20, grid_w=25, n_blocks=7, keep_monolithic=1)]  # with a shared queue
LABELS = [0, 1, 2, 3, 2, 3]


def unordered(log):
    """The launches, and the pairs of them on one scratch of which the earlier need not have ended when the later one starts."""
    launches, done, before, events, pairs = [], set(), {}, {}, []  # before: what comes first on a stream, by its waits
    for entry in log.decode().split():
        stream, _, what = entry[1:].partition(":")
        past = done | before.get(stream, set()) | {i for i, (s, _) in enumerate(launches) if s == stream}
        if entry[0] == "E":
            events[what] = past
        elif entry[0] == "Y":
            done = past
        elif entry[0] == "W":
            before[stream] = before.get(stream, set()) | events[what]
        elif entry[0] == "L" and ("attn_kernel" in what or "combine_kernel" in what):
            scratch = what.partition("@")[2]
            pairs += [(i, len(launches)) for i, (_, other) in enumerate(launches) if other == scratch and i not in past]
            launches.append((stream, scratch))
    return launches, pairs


def ready(fake, cfg):
    ctx = fake.context(**cfg)
    assert ctx.append(cfg["n_blocks"]) == 0 and ctx.split(LABELS[:cfg["n_heads"]]) == 0
    assert ctx.attend(11) == 0 and ctx.full_attend(11) == 0  # both lists are uploaded
    fake.clear_log()
    return ctx


@pytest.mark.parametrize("cfg", SIZES)
def test_calls_on_changing_streams_follow_one_another(cfg):
    fake = FakeLibrary()
    ctx = ready(fake, cfg)
    for stream in (11, 12, 12, 11, 13, 0, 12, 11, 11, 12, 13, 13, 0, 11):
        assert ctx.attend(stream) == 0 and ctx.full_attend(stream) == 0
    launches, pairs = unordered(fake.log())
    assert len(launches) == 14 * 4 and not pairs
    assert len({scratch for _, scratch in launches}) <= 5  # four sets, the first of which may have grown
    assert b"S " not in fake.log()  # nothing waits for the device
    used = fake.used()
    for i in range(40):
        assert ctx.attend(11 + i % 3) == 0 and ctx.full_attend(11 + i % 2) == 0
    assert fake.used() == used
    assert ctx.destroy() == 0 and fake.lib.headcast_release_memory() == 0 and fake.used() == 0


def test_streams_may_change_beside_the_capture_of_another():
    fake = FakeLibrary()
    ctx = ready(fake, SIZES[0])
    fake.capture(RELAXED, 99)
    for stream in (12, 13, 12, 14, 12):
        assert ctx.attend(stream) == 0
    assert not fake.capture_invalidated() and not unordered(fake.log())[1]


@pytest.mark.parametrize("cfg", SIZES)
def test_calls_on_one_stream_record_and_wait_for_nothing(cfg):
    fake = FakeLibrary()
    ctx = ready(fake, cfg)
    for _ in range(4):
        assert ctx.attend(11) == 0 and ctx.full_attend(11) == 0
    assert all(entry.startswith("L") for entry in fake.log().decode().split())


def test_a_captured_call_records_and_waits_for_nothing():
    fake = FakeLibrary()
    ctx = ready(fake, SIZES[0])
    for stream in (12, 11, 12, 11, 12):
        assert ctx.attend(stream) == 0
    fake.clear_log()
    fake.capture(RELAXED, 21)
    assert ctx.attend(21) == 0
    assert all(entry.startswith("L") for entry in fake.log().decode().split())
    fake.capture(0, None)
    assert ctx.attend(12) == 0 and ctx.attend(11) == 0
    assert "W11:" in fake.log().decode() and "W12:" not in fake.log().decode()
