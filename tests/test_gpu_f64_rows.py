"""FP64 rows of every envelope length against the FP64 oracle: compile-time shapes
for bisquare bands, the runtime engine for window tables and dense tiles; few rows
(partly filled blocks) and row selections.

Tolerances: 1.1e-16 sqrt(log2 M) <= 4e-16 a transform, window and oracle as much
again; 1e-14 leaves a factor of ten."""
import numpy as np
import pytest

from oracle import qtam_oracle as O
from paper_2603_29785_gb300 import qtam, synth

from .test_gpu_row_lengths import LENGTHS, geometry, rel

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def check(M, **kw):
    g = geometry(M)
    p = qtam.Plan(device=0, compute="f64", **g, **kw)
    o = O.geometry(*list(g.values())[:6], max_window_hz=g["max_window_hz"], n_out=M, **kw)
    B = 3
    x = np.stack([synth.white(10 * M + b, p.N) for b in range(B)]).astype(np.float64)
    X = np.stack([O.spectrum(v) for v in x])
    y = p.envelopes(torch.from_numpy(X).cuda()).cpu().numpy()
    S = synth.rng(M).standard_normal((B, o.P, o.K, M, 2))
    src = torch.view_as_complex(torch.from_numpy(S)).cuda()
    for mask, planes in ((0, None), (2, [1])):
        A = p.accumulate(src, plane_mask=mask).cpu().numpy()
        for b in range(B):
            assert rel(y[b], O.forward(o, x[b])) < 1e-14, (M, b)
            assert rel(A[b], O.accumulate(o, S[b, ..., 0] + 1j * S[b, ..., 1], planes=planes)) < 1e-14, (M, b, mask)


@pytest.mark.parametrize("part", range(2))
def test_every_length(part):
    for M in LENGTHS[part::2]:
        check(M)


def test_other_modes():
    for M in (81, 250, 1125, 4096):
        check(M, window=("hann", "bisquare"), window_param=(0.0, 0.0))
        check(M, remodulate=True)
