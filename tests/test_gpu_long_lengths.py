"""The long real FFT and its inverse at segment lengths N = 2 * 2^a 3^b 5^c, so
that every compile-time pass length and ragged groups of rows and columns occur
(N up to 2^20), against FP64 transforms.

Tolerances: FP32 arithmetic, rms relative error ~ 6e-8 sqrt(log2 N) <= 3e-7 per
transform; table roundings (1/P, twiddles) at most double it, so 1e-6."""
import numpy as np
import pytest

from paper_2603_29785_gb300 import qtam

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

HALVES = sorted(2 ** a * 3 ** b * 5 ** c for a in range(20) for b in range(13) for c in range(9)
                if 64 <= 2 ** a * 3 ** b * 5 ** c <= 1 << 19)
GROUPS = 16


def rel(a, b):
    return float(torch.linalg.norm(a - b) / torch.linalg.norm(b))


def plan(N, compute):
    T = 16.0                                   # bins 1/16 Hz wide, windows of at most 4 Hz
    fs = N / T
    f_max = 0.45 * fs
    return qtam.Plan(fs, N, (4.0,), min(1.0, 0.5 * f_max), f_max, 3, max_window_hz=min(4.0, 0.1 * fs), compute=compute,
                     device=0)


def check(N, compute, tol):
    p = plan(N, compute)
    B = 2
    gen = torch.Generator(device="cuda").manual_seed(N)
    x = torch.randn((B, N), generator=gen, device="cuda", dtype=p.real_dtype())
    assert rel(p.spectrum(x).to(torch.complex128), torch.fft.rfft(x.double())) < tol, N
    P = torch.from_numpy(np.asarray(p.frame_operator())).cuda()
    A = torch.randn((B, N // 2 + 1, 2), generator=gen, device="cuda", dtype=p.real_dtype())
    Xh = torch.view_as_complex(A.double())
    tau = 0.0 if compute == "f64" else 1e-6
    keep = (P > 0) & (P >= tau * P.max())
    Xh = Xh * torch.where(keep, 1 / P, torch.zeros_like(P))
    Xh.imag[:, 0] = 0
    Xh.imag[:, -1] = 0
    out = p.synthesize(torch.view_as_complex(A)).double()
    assert rel(out, torch.fft.irfft(Xh, n=N)) < tol, N


@pytest.mark.parametrize("group", range(GROUPS))
def test_lengths_f32(group):
    for n in HALVES[group::GROUPS]:
        check(2 * n, "f32", 1e-6)


@pytest.mark.parametrize("group", range(4))
def test_lengths_f64(group):
    """Every eighth length in FP64: 1.1e-16 sqrt(log2 N) <= 5e-16 a transform, tables as much again, FP64
    reference alike; 1e-14 leaves a factor of five."""
    for n in HALVES[2 * group::32]:
        check(2 * n, "f64", 1e-14)
