"""Branches of a recorded pass (detector._Lanes): which calls wait for which, on host tensors with fake streams."""
import pytest
import torch

from paper_2609_10632_b200 import detector


@pytest.mark.parametrize("a,b,conflict", [
    ((0, 8), (8, 24), False), ((0, 8), (0, 8), True), ((0, 16), (8, 24), True), ((24, 32), (0, 24), False), ((0, 32), (16, 24), True),
], ids=["beside", "same", "overlapping", "last and rest", "whole and part"])
def test_channel_ranges_of_one_buffer(a, b, conflict):
    buf = torch.zeros(2, 3, 5, 32, dtype=torch.bfloat16)
    spans = [detector._span(buf[..., lo:hi]) for lo, hi in (a, b)]
    assert detector._overlap(*spans) is conflict and detector._overlap(*spans[::-1]) is conflict


def test_other_objects_and_pieces_of_a_flat_buffer():
    flat, plan = torch.zeros(64), object()
    part = [detector._span(flat[i:j]) for i, j in ((0, 32), (32, 64), (31, 33))]
    assert not detector._overlap(part[0], part[1]) and detector._overlap(part[0], part[2]) and detector._overlap(part[2], part[1])
    assert detector._overlap(detector._span(plan), detector._span(plan)) and not detector._overlap(detector._span(plan), part[0])


def test_branches_keep_the_order_of_conflicting_calls(monkeypatch):
    class Event:
        def record(self, stream):
            self.covers = set(stream.done)

    class Stream:
        def __init__(self, device=None):
            self.done = set()

        def wait_event(self, event):
            self.done |= event.covers

    monkeypatch.setattr(detector.torch.cuda, "Event", Event)
    monkeypatch.setattr(detector.torch.cuda, "Stream", Stream)
    t = [torch.zeros(4) for _ in range(6)]
    #        reads  writes: a chain, two branches off it that both add to t[4], what needs both, and a call of its own
    calls = [((0,), (1,)), ((1,), (2,)), ((1,), (3,)), ((2,), (4,)), ((3,), (4,)), ((4,), (0,)), ((), (5,))]
    before = [set(), {0}, {0}, {0, 1}, {0, 1, 2, 3}, {0, 1, 2, 3, 4}, set()]
    main = Stream()
    lanes = detector._Lanes(main, None, [])
    for i, (reads, writes) in enumerate(calls):
        stream = lanes.enter([t[k] for k in reads] + [None], [t[k] for k in writes])
        assert stream.done == before[i]  # everything it has a conflict with, and nothing else
        stream.done.add(i)
    lanes.finish()
    assert main.done == set(range(len(calls))) and len(lanes.streams) == 3


def test_no_collection_while_any_recording_is_open():
    import gc
    import threading

    assert gc.isenabled()
    block, opened, leave = detector._NoCollection(), threading.Event(), threading.Event()

    def other():
        with block:
            opened.set()
            leave.wait(10)

    thread = threading.Thread(target=other)
    with block:
        thread.start()
        opened.wait(10)
        assert not gc.isenabled()
    assert not gc.isenabled()  # the other thread's recording goes on
    leave.set()
    thread.join()
    assert gc.isenabled()
    gc.disable()
    try:
        with block:
            pass
        assert not gc.isenabled()  # left as it was found
    finally:
        gc.enable()
