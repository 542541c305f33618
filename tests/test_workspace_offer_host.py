"""The workspace that an FP64 call takes when there is room (Handle.offer_workspace), on a
fake device: no more than a quarter of the free memory, nothing under a capture, and
after a refusal or a failed allocation no further attempt for the next calls that ask
for as much."""
import contextlib

import pytest
import torch

from paper_2504_13821_gb300 import _binding


class Fake(_binding.Handle):
    """A handle without a library behind it that counts its allocations."""

    def __init__(self, fails=False):
        self._h, self.device = None, torch.device("cuda", 0)
        self._ws, self._ws_bytes = None, 0
        self._declined, self._declined_calls = float("inf"), 0
        self.fails, self.attempts = fails, []

    def ensure_workspace(self, nbytes):
        self.attempts.append(nbytes)
        if self.fails:
            raise torch.cuda.OutOfMemoryError("fake")
        self._ws_bytes = nbytes


@pytest.fixture
def device(monkeypatch):
    state = {"free": 1000, "cached": 0, "capturing": False, "looks": 0}

    def mem_get_info(_):
        state["looks"] += 1
        return state["free"], 10000
    none = lambda *a, **k: contextlib.nullcontext()
    for name, f in (("device", none), ("stream", none), ("mem_get_info", mem_get_info),
                    ("memory_reserved", lambda d: state["cached"]),
                    ("memory_allocated", lambda d: 0),
                    ("is_current_stream_capturing", lambda: state["capturing"])):
        monkeypatch.setattr(torch.cuda, name, f)
    return state


def test_takes_a_quarter_at_most(device):
    h = Fake()
    h.offer_workspace(250)
    h.offer_workspace(250)
    assert h.attempts == [250]
    h = Fake()
    h.offer_workspace(251)
    assert h.attempts == []
    device["cached"] = 400
    h = Fake()
    h.offer_workspace(350)
    assert h.attempts == [350]


def test_nothing_under_a_capture(device):
    h = Fake()
    device["capturing"] = True
    h.offer_workspace(10)
    assert h.attempts == []
    device["capturing"] = False
    h.offer_workspace(10)
    assert h.attempts == [10]


@pytest.mark.parametrize("fails", [True, False])
def test_a_refusal_is_not_tried_again_at_once(device, fails):
    h = Fake(fails)
    size = 100 if fails else 300
    for _ in range(h.RETRY + 1):
        h.offer_workspace(size)
    assert device["looks"] == 1 and len(h.attempts) == fails
    h.offer_workspace(size)
    assert device["looks"] == 2
    h.offer_workspace(50)                         # a smaller size is another question
    assert h.attempts[-1] == 50 and device["looks"] == 3
