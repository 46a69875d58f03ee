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


def test_growth(plan):
    a, _ = plan.workspace(1, 5)
    b, nb = plan.workspace(9, 5)
    assert b is not a and nb >= qtam.qtam_workspace_size(plan.handle, 9)
    assert plan.workspace(1, 5)[0] is b


def test_scratch_lives_as_long_as_the_plan(plan):
    """A graph captured by a thread that has ended, or before many other streams were used, still replays on it."""
    import weakref
    refs = [weakref.ref(plan.workspace(1, 5)[0])]
    t = threading.Thread(target=lambda: refs.append(weakref.ref(plan.workspace(1, 6)[0])))
    t.start()
    t.join()
    for s in range(100, 200):
        plan.workspace(1, s)
    assert all(r() is not None for r in refs)


class FakeTensor:
    """What the argument checks read of a device tensor (of a host-only plan's device, -1)."""
    is_cuda = True

    def __init__(self, shape, dtype):
        self.shape, self.dtype = shape, dtype

    def get_device(self):
        return -1

    def is_contiguous(self):
        return True

    def dim(self):
        return len(self.shape)

    def data_ptr(self):
        return 256


def test_single_tile_output_holds_the_batch(monkeypatch):
    """The kernels write B segments: an output with fewer is refused before they are launched."""
    torch = pytest.importorskip("torch")
    monkeypatch.setattr(qtam.Plan, "_scratch", lambda self, nbytes, st: FakeTensor((nbytes,), torch.uint8), raising=False)
    monkeypatch.setattr(FakeTensor, "numel", lambda self: self.shape[0], raising=False)
    monkeypatch.setattr(qtam, "_stream", lambda s: s or 0)
    p = qtam.Plan(64.0, 256, (3.0,), 2.0, 31.0, 5, n_out=135, stopband_eps=1e-3, device=-1)
    y = FakeTensor((3, p.P, p.K, p.M), torch.complex64)
    with pytest.raises(ValueError, match="batch sizes differ"):
        p.inverse_single_tile(y, 0, 1, x=FakeTensor((2, p.N), torch.float32))
    with pytest.raises(qtam.QtamError) as e:           # the right size reaches the library, which has no device
        p.inverse_single_tile(y, 0, 1, x=FakeTensor((3, p.N), torch.float32))
    assert e.value.status == 8


def test_negative_batch_is_refused(plan):
    for _ in range(2):
        with pytest.raises(qtam.QtamError) as e:
            plan.workspace(-1, 11)
        assert e.value.status == 1


def test_the_binding_loads_without_pytorch():
    """Geometry and planning on the host need no device memory, so no import of PyTorch (seconds)."""
    import subprocess
    import sys
    code = ("import sys; from paper_2603_29785_gb300 import qtam; p = qtam.Plan(4096.0, 16384, (8.0,), 20.0, 1024.0, 16, "
            "device=-1); p.frame_operator(); assert 'torch' not in sys.modules")
    subprocess.run([sys.executable, "-c", code], check=True, cwd=qtam._build.ROOT)
