"""The accumulator is cleared whatever its alignment and size: odd bin counts, one
segment and many, starting on 8 but not on 16 bytes."""
import pytest

from paper_2603_29785_gb300 import qtam

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("compute", ["f32", "f64"])
@pytest.mark.parametrize("N,B", [(64, 1), (1000, 1), (1024, 3), (16384, 700)])
@pytest.mark.parametrize("offset", [0, 1])
def test_accumulate_clears(compute, N, B, offset):
    p = qtam.Plan(64.0, N, (4.0,), 8.0, 28.0, 3, max_window_hz=8.0, compute=compute, device=0)
    A = torch.full((B * p.Nr + 2 + offset,), 7.0 + 3.0j, device="cuda", dtype=p.complex_dtype())
    y = torch.zeros((B, p.P, p.K, p.M), device="cuda", dtype=p.complex_dtype())
    qtam.qtam_stage_accumulate(p.handle, y, B, 0, A[offset:])
    assert not A[offset:offset + B * p.Nr].any()
    assert (A[:offset] == 7.0 + 3.0j).all() and (A[offset + B * p.Nr:] == 7.0 + 3.0j).all()
