"""Plane metrics at the edges of their block split, and the plane choice."""
import pytest

from paper_2603_29785_gb300 import qtam

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("B,N,K", [(1, 1024, 3), (3, 4096, 7), (700, 1024, 3)])
def test_plane_metrics_split_and_choice(B, N, K):
    """Energies and peaks of few and many (segment, plane) pairs (blocks of one
    to 64 parts) against FP64 sums of the same envelopes, FP32 partials of at
    most 8 terms: 5e-7; the chosen planes, with ties, infinities and NaN."""
    p = qtam.Plan(256.0, N, (4.0, 8.0, 16.0, 23.0), 4.0, 100.0, K, device=0)
    gen = torch.Generator(device="cuda").manual_seed(B)
    y = torch.randn((B, p.P, p.K, p.M), generator=gen, device="cuda", dtype=torch.complex64)
    y[:, 2] = y[:, 1]                                  # ties: the first plane wins
    if B > 2:
        y[1, 3, 0, 0] = float("inf")
        y[2, 1, 0, 0] = float("nan")
    energy, peak, best_e, best_p = p.plane_metrics(y)
    a2 = torch.view_as_real(y).double().square().sum(-1)
    e, pk = a2.sum((2, 3)), a2.amax((2, 3))
    fin = torch.isfinite(e)
    assert torch.equal(torch.isfinite(energy), fin)
    assert ((energy - e).abs()[fin] <= 5e-7 * e[fin]).all()
    assert ((peak - pk).abs()[fin] <= 3e-7 * pk[fin]).all()
    assert torch.equal(best_e, energy.argmax(dim=1)) and torch.equal(best_p, peak.argmax(dim=1))
    assert best_e.dtype == torch.int64 and best_p.shape == (B,)
