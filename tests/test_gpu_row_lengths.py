"""The row kernels of every envelope length (2^a 3^b 5^c from 2 to 7680, and
8192): analysis and accumulation against the FP64 oracle with windows as wide
as the length allows, an odd number of rows (partly filled blocks), and the
storage, window and dense-mode options on a spread of lengths.

Tolerances: FP32 arithmetic, rms relative error ~ 6e-8 sqrt(log2 M) <= 3e-7 per
transform plus the window's 2e-7, so 1e-6; 16-bit storage adds 2^-9 (BF16) or
2^-12 (FP16) per component."""
import numpy as np
import pytest

from oracle import qtam_oracle as O
from paper_2603_29785_gb300 import qtam, synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _smooth(m):
    for p in (2, 3, 5):
        while m % p == 0:
            m //= p
    return m == 1


LENGTHS = [m for m in range(3, 7681) if _smooth(m)] + [8192]


def rel(a, b):
    return np.linalg.norm(a - b) / np.linalg.norm(b)


def geometry(M, **kw):
    """fs, N, planes ... with h = (M - 1) // 2 on the clamped rows"""
    N = 1 << max(8, (2 * M - 1).bit_length())
    fs = 64.0
    hz = 2 * ((M - 1) // 2) / (N / fs)
    return dict(sample_rate=fs, length=N, qs=(1.5, 20.0), f_min=2.0, f_max=31.0, rows_per_plane=5, max_window_hz=hz,
                n_out=M, **kw)


def check(M, fwd_tol, acc_tol, **kw):
    g = geometry(M)
    opts = {k: v for k, v in kw.items() if k != "envelope"}
    p = qtam.Plan(device=0, **g, **kw)
    o = O.geometry(*list(g.values())[:6], max_window_hz=g["max_window_hz"], n_out=M, **opts)
    assert p.M == M
    B = 3
    x = np.stack([synth.white(10 * M + b, p.N) for b in range(B)])
    X = [O.spectrum(v) for v in x]
    y = p.envelopes(torch.from_numpy(np.stack(X).astype(np.complex64)).cuda())
    Y = y.float().cpu().numpy() if p.envelope != "f32" else torch.view_as_real(y).cpu().numpy()
    Y = Y[..., 0].astype(np.float64) + 1j * Y[..., 1]
    for b in range(B):
        ref = O.forward(o, x[b])
        assert rel(Y[b], ref) < fwd_tol, (M, b, rel(Y[b], ref))
    r = synth.rng(M)
    S = r.standard_normal((B, o.P, o.K, M, 2)).astype(np.float32)
    t = torch.from_numpy(S)
    if p.envelope != "f32":
        t = t.to(y.dtype)
        S = t.float().numpy()
    src = t.cuda() if p.envelope != "f32" else torch.view_as_complex(t).cuda()
    for mask, planes in ((0, None), (2, [1])):
        A = p.accumulate(src, plane_mask=mask).cpu().numpy().astype(np.complex128)
        for b in range(B):
            ref = O.accumulate(o, S[b, ..., 0].astype(np.float64) + 1j * S[b, ..., 1], planes=planes)
            assert rel(A[b], ref) < acc_tol, (M, b, mask, rel(A[b], ref))


@pytest.mark.parametrize("part", range(4))
def test_every_length(part):
    for M in LENGTHS[part::4]:
        check(M, 1e-6, 1e-6)


SPREAD = [3, 16, 50, 81, 128, 270, 640, 675, 1000, 1125, 2025, 2250, 3600, 4096, 5625, 6750, 7680, 8192]


@pytest.mark.parametrize("env,tol", [("bf16", 4e-3), ("f16", 5e-4)])
def test_16_bit_storage(env, tol):
    for M in SPREAD:
        check(M, tol, 1e-6, envelope=env)


@pytest.mark.parametrize("env,tol", [("f32", 1e-6), ("bf16", 4e-3)])
def test_window_tables(env, tol):
    for M in SPREAD:
        check(M, tol, 1e-6, envelope=env, window=("hann", "bisquare"), window_param=(0.0, 0.0))


@pytest.mark.parametrize("eps,remod", [(1e-3, False), (1e-3, True), (0.0, True)])
def test_dense_options(eps, remod):
    for M in (135, 144, 150, 600, 1080, 1125, 2160, 4374):
        N = 1 << ((M - 1).bit_length())          # M >= N / 2 + 1: tiles may span the spectrum
        kw = dict(stopband_eps=eps, remodulate=remod)
        p = qtam.Plan(64.0, N, (3.0, 20.0), 2.0, 31.0, 5, n_out=M, device=0, **kw)
        o = O.geometry(64.0, N, (3.0, 20.0), 2.0, 31.0, 5, n_out=M, **kw)
        x = np.stack([synth.white(M + b, N) for b in range(3)]).astype(np.float32)
        y = p.forward(torch.from_numpy(x).cuda())
        Y = y.cpu().numpy().astype(np.complex128)
        xh = p.inverse(y).cpu().numpy().astype(np.float64)
        for b in range(3):
            assert rel(Y[b], O.forward(o, x[b].astype(np.float64))) < 1e-6, M
            assert rel(xh[b], O.projection(o, x[b].astype(np.float64), tau=p.info["p_floor_rel"])) < 1e-5, M
        if eps > 0:
            xs = p.inverse_single_tile(y, 1, 2).cpu().numpy()
            assert rel(xs, x) < 1e-3, M      # the division lifts FP32 rounding by about sqrt(L / M) / eps
