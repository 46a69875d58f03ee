"""A launch that CUDA refuses is reported by the call that made it, and by no later one."""
import ctypes

import pytest

from paper_2603_29785_gb300 import qtam

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("N", [65536, 24576, 2 * 8 * 2048])     # static columns, compile-time columns, few columns
def test_a_refused_launch_is_reported_once(N):
    """Launches into a stream capture that a forbidden call has ended are refused, with
    nothing queued; the same calls after the capture are good ones."""
    cu = ctypes.CDLL("libcuda.so.1")
    p = qtam.Plan(4096.0, N, (8.0,), 20.0, 1024.0, 16, device=0)
    x = torch.randn((2, N), device="cuda")
    y = p.envelope_tensor(2)
    s = torch.cuda.Stream()
    p.forward(x, y, stream=s)
    A = p.accumulate(y, stream=s)
    p.synthesize(A, stream=s)
    torch.cuda.synchronize()
    want = y.clone()
    x2, gain = torch.empty_like(x), torch.ones((2, p.P, p.K), device="cuda")
    torch.cuda.synchronize()
    for call in (lambda: p.forward(x, y, stream=s), lambda: p.inverse(y, x=x2, stream=s),
                 lambda: p.scale_rows(y, gain, stream=s)):
        h = ctypes.c_void_p(s.cuda_stream)
        assert cu.cuStreamBeginCapture_v2(h, 2) == 0            # relaxed
        assert cu.cuStreamSynchronize(h) != 0                   # not allowed: the capture is invalid now
        with pytest.raises(qtam.QtamError) as e:
            call()
        assert e.value.status == 6
        g = ctypes.c_void_p()
        assert cu.cuStreamEndCapture(h, ctypes.byref(g)) != 0 and not g.value
        again = p.forward(x, stream=s)                          # raises nothing
        s.synchronize()
        assert torch.equal(again, want)
