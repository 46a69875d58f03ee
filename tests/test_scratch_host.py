"""Which scratch buffer a call gets: calls that may run at the same time never share one."""
import threading

import pytest

from paper_2603_29785_gb300 import qtam


class Buffer:
    def __init__(self, nbytes, stream):
        self.nbytes, self.stream = nbytes, stream

    def numel(self):
        return self.nbytes


@pytest.fixture
def plan(monkeypatch):
    monkeypatch.setattr(qtam.Plan, "_scratch", lambda self, nbytes, st: Buffer(nbytes, st), raising=False)
    return qtam.Plan(4096.0, 16384, (8.0,), 20.0, 1024.0, 16, device=-1)


def test_each_stream_and_thread_has_its_own(plan):
    a, na = plan.workspace(4, 11)
    b, _ = plan.workspace(4, 12)
    assert a is not b and (a.stream, b.stream) == (11, 12)
    assert plan.workspace(3, 11)[0] is a and plan.workspace(4, 12)[0] is b     # kept while it is large enough
    assert na == a.numel() == qtam.qtam_workspace_size(plan.handle, 4)
    other = []
    t = threading.Thread(target=lambda: other.append(plan.workspace(4, 11)[0]))
    t.start()
    t.join()
    assert other[0] is not a and other[0].stream == 11
    assert plan.workspace(4, 11)[0] is a


def test_growth_and_bound(plan):
    a, _ = plan.workspace(1, 5)
    b, nb = plan.workspace(9, 5)
    assert b is not a and nb >= qtam.qtam_workspace_size(plan.handle, 9)
    assert plan.workspace(1, 5)[0] is b
    first, _ = plan.workspace(1, 100)
    for s in range(101, 100 + plan.MAX_SCRATCH):
        plan.workspace(1, s)
    assert plan.workspace(1, 100)[0] is first and plan.workspace(1, 5)[0] is not b     # the oldest went first
    assert len(plan._ws.by_stream) == plan.MAX_SCRATCH
