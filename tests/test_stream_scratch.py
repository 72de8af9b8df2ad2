"""Which scratch buffer a call takes, on the host alone (no GPU): calls on two
streams never share one, what is kept is bounded, and another stream's buffer
outlives a call of another size."""
import threading
import time

import pytest
import torch

from paper_2510_07729_gb300 import sop


class FakeLib:
    """Records the workspace of every bake; enqueuing takes a while."""

    def __init__(self):
        self.seen, self.inside, self.overlap = [], 0, False

    def sop_bake_workspace_bytes(self, n, P, R):
        return 1024 + n

    def sop_surrogate_workspace_bytes(self, n, P, R):
        return 1024 + n

    def sop_bake(self, g, d, bp, ws, nbytes, stream):
        self.inside += 1
        self.overlap |= self.inside > 1
        time.sleep(0.01)
        self.seen.append((stream, ws))
        self.inside -= 1
        return 0


@pytest.fixture
def host(monkeypatch):
    lib = FakeLib()
    here = threading.local()
    monkeypatch.setattr(sop, "load", lambda: lib)
    monkeypatch.setattr(sop, "_ptr", lambda t: None if t is None else t.data_ptr())
    monkeypatch.setattr(sop, "_stream", lambda: getattr(here, "stream", 0))
    monkeypatch.setattr(sop, "_capturing", lambda: getattr(here, "capturing", False), raising=False)
    monkeypatch.setattr(sop, "_bake_ws", type(sop._bake_ws)())
    return lib, here


def scene(n):
    g = dict(mean=torch.zeros(n, 3), scale=torch.ones(n, 3), quat=torch.ones(n, 4), opacity=torch.ones(n),
             rgb=torch.ones(n, 3))
    return g, sop.make_atlas(torch.zeros(2, 3), 4)


def test_streams_do_not_share_a_bake_workspace(host):
    lib, here = host
    g, at = scene(5)
    for here.stream in (11, 12, 11, 12):
        sop.bake(g, at)
    a, b = lib.seen[0][1], lib.seen[1][1]
    assert a != b and [w for _, w in lib.seen] == [a, b, a, b]


def test_another_size_leaves_the_other_streams_buffer(host):
    lib, here = host
    here.stream = 11
    sop.bake(*scene(5))
    kept = lib.seen[-1][1]
    here.stream = 12
    sop.bake(*scene(7))
    here.stream = 11
    sop.bake(*scene(5))
    assert lib.seen[-1][1] == kept


def test_kept_buffers_are_bounded(host):
    lib, here = host
    for here.stream in range(50):
        sop.bake(*scene(3))
    assert len(sop._bake_ws._kept) == 4


def test_a_captured_bake_keeps_nothing(host):
    lib, here = host
    here.capturing = True
    sop.bake(*scene(3))
    assert len(lib.seen) == 1 and not sop._bake_ws._kept


def test_threads_on_one_stream_enqueue_in_turn(host):
    lib, here = host
    g, at = scene(4)
    threads = [threading.Thread(target=lambda: [sop.bake(g, at) for _ in range(3)]) for _ in range(4)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert len(lib.seen) == 12 and len({w for _, w in lib.seen}) == 1 and not lib.overlap
