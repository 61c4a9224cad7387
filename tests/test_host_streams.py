"""headcast_attend_host on several streams, on a CUDA runtime made for tests: all calls of a context go through one pair of staging
buffers, so the copies and launches of a call come after those of the call before it, whichever stream either is on."""
import ctypes as C

import pytest

from fake_cuda import RELAXED, FakeLibrary

# blocks of 0.1 and 4.5 MiB of queries: copied, attended and copied back as one, and in four stages
SIZES = [dict(n_heads=4, head_dim=64, grid_h=8, grid_w=8, n_blocks=3), dict(n_heads=6, head_dim=128, grid_h=32, grid_w=32, n_blocks=3)]


def unordered(log):
    """(number of calls, pairs of calls of which the earlier need not have ended when the later one's first copy starts).  A call's
    copies and launches end at the marker that the test writes behind it."""
    ops, done, before, events, pairs, call = [], set(), {}, {}, [], 0  # ops: (stream, call)
    for entry in log.split():
        if entry == "|":
            call += 1
            continue
        stream, _, what = entry[1:].partition(":")
        past = done | before.get(stream, set()) | {i for i, (s, _) in enumerate(ops) if s == stream}
        if entry[0] == "E":
            events[what] = past
        elif entry[0] == "Y":
            done = past
        elif entry[0] == "W":
            before[stream] = before.get(stream, set()) | events.get(what, set())
        elif entry[0] in "HDL":
            pairs += [(c, call) for i, (_, c) in enumerate(ops) if c < call and i not in past]
            ops.append((stream, call))
    return call, sorted(set(pairs))


class Caller:
    def __init__(self, cfg, labels=(0, 1, 2, 3, 2, 3)):
        self.fake = FakeLibrary()
        self.ctx = self.fake.context(**cfg)
        labels = list(labels)[:cfg["n_heads"]]
        assert self.ctx.append(3) == 0 and self.ctx.split(labels) == 0
        bytes_ = 2 * 3 * cfg["grid_h"] * cfg["grid_w"] * cfg["n_heads"] * cfg["head_dim"]
        self.buffers = [C.create_string_buffer(bytes_) for _ in range(2)]
        self.log = ""

    def attend(self, stream):
        self.fake.clear_log()
        rc = self.fake.lib.headcast_attend_host(self.ctx.ptr, *(C.addressof(b) for b in self.buffers), stream)
        self.log += self.fake.log().decode() + " | "
        return rc


@pytest.mark.parametrize("cfg", SIZES)
def test_calls_on_changing_streams_follow_one_another(cfg):
    caller = Caller(cfg)
    for stream in (11, 11):
        assert caller.attend(stream) == 0
    caller.log = ""  # the lists are uploaded: nothing waits on the host any more
    for stream in (11, 12, 11, 13, 0, 12, 12, 11, 14, 13):
        assert caller.attend(stream) == 0
    assert unordered(caller.log) == (10, []) and "Y" not in caller.log and "S" not in caller.log.split()
    assert caller.ctx.destroy() == 0 and caller.fake.lib.headcast_release_memory() == 0 and caller.fake.used() == 0


@pytest.mark.parametrize("cfg", SIZES)
def test_calls_on_one_stream_wait_for_no_earlier_call(cfg):
    caller = Caller(cfg)
    for _ in range(4):
        assert caller.attend(11) == 0
    assert unordered(caller.log) == (4, [])
    if cfg is SIZES[0]:
        assert "W" not in caller.log


@pytest.mark.parametrize("cfg", SIZES)
def test_no_event_passes_between_a_captured_call_and_others(cfg):
    caller = Caller(cfg)
    assert caller.attend(11) == 0 and caller.attend(12) == 0
    caller.log = ""
    caller.fake.capture(RELAXED, 21)
    assert caller.attend(21) == 0
    captured, caller.log = caller.log.split(), ""
    caller.fake.capture(0, None)
    assert caller.attend(12) == 0 and caller.attend(11) == 0
    recorded, seen = set(), set()
    for log, known in ((captured, seen), (caller.log.split(), recorded)):  # every wait is for an event of its own side
        for entry in log:
            event = entry.partition(":")[2]
            if entry[0] == "E":
                known.add(event)
            elif entry[0] == "W" and log is captured:
                assert event in known
            elif entry[0] == "W":
                assert event in known or event not in seen
    assert unordered(caller.log) == (2, [])


@pytest.mark.parametrize("cfg", SIZES)
def test_a_call_that_failed_half_way_is_waited_for_too(cfg):
    caller = Caller(cfg)
    assert caller.fake.lib.headcast_release_memory() == 0
    caller.fake.capacity_left(2 << 17 if cfg is SIZES[0] else 12 << 20)  # room for the two staging buffers, not for a list
    caller.log = ""
    assert caller.attend(11) == -4 and any(entry[0] == "H" for entry in caller.log.split())
    caller.fake.capacity_left(1 << 40)
    assert caller.attend(12) == 0
    assert unordered(caller.log) == (2, [])


@pytest.mark.parametrize("labels,grid_h,grid_w,as_one", [
    ([3] * 12, 9, 9, True),                  # one stage: up to 256 rows of Global heads
    ([3] * 12, 16, 28, False),               # two halves of the Global heads' rows, one copy each
    ([2] * 12, 16, 28, True),                # one stage
    ([0, 1] * 6, 16, 28, True),
    ([2] * 3 + [3] * 3, 10, 17, True),       # three copies: up to 768 KB, 512 rows of six heads
    ([2] * 3 + [3] * 3, 9, 19, False),
    ([2, 3] * 6, 16, 28, True),              # eighteen copies
    ([2, 3] * 6, 19, 24, False),             # more than 4 MiB
])
def test_blocks_are_cut_where_the_copies_of_the_stages_are_few(labels, grid_h, grid_w, as_one):
    caller = Caller(dict(n_heads=len(labels), head_dim=128, grid_h=grid_h, grid_w=grid_w, n_blocks=3), labels)
    assert caller.attend(11) == 0
    caller.log = ""
    assert caller.attend(11) == 0
    assert (sum(entry[0] == "H" for entry in caller.log.split()) == 1 and "E11" in caller.log and "W" not in caller.log) == as_one
