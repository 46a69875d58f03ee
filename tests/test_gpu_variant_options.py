"""Registered row variants with the options a tuner may choose them for: 16-bit
storage, window tables (a bisquare plane among them) and dense tiles.  Plans run the
kernels of their own length until one is selected, so each is selected here.

Tolerances as for the length's own kernels: FP32 arithmetic 1e-6 a transform, 16-bit
storage 2^-9 (BF16) or 2^-12 (FP16) a component, 1e-5 for a whole inverse."""
import numpy as np
import pytest

from oracle import qtam_oracle as O
from paper_2603_29785_gb300 import qtam, synth

from .test_gpu_row_lengths import geometry, rel

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

LENGTHS = (75, 150, 300, 500, 600, 1200, 2400, 4800, 8192)
STORED = {"f32": 1e-6, "bf16": 4e-3, "f16": 5e-4}


def registered(p):
    ids = [v for v in qtam.qtam_plan_variants(p.handle) if v != -1]
    assert ids
    for v in ids:
        qtam.qtam_plan_set_variant(p.handle, v)
        assert qtam.qtam_plan_running_variant(p.handle) == v
        yield qtam.qtam_variant_describe(v)["name"]


def values(y):
    a = (y if y.dtype.is_complex is False else torch.view_as_real(y)).cpu().double().numpy()
    return a[..., 0] + 1j * a[..., 1]


@pytest.mark.parametrize("M", LENGTHS)
@pytest.mark.parametrize("env,kw", [("bf16", {}), ("f16", {}),
                                    ("f32", dict(window=("hann", "bisquare"), window_param=(0.0, 0.0)))])
def test_storage_and_tables(M, env, kw):
    g = geometry(M)
    p = qtam.Plan(device=0, envelope=env, **g, **kw)
    o = O.geometry(*list(g.values())[:6], max_window_hz=g["max_window_hz"], n_out=M, **kw)
    B = 3
    x = np.stack([synth.white(10 * M + b, p.N) for b in range(B)])
    X = torch.from_numpy(np.stack([O.spectrum(v) for v in x]).astype(np.complex64)).cuda()
    refs = [O.forward(o, v) for v in x]
    S = torch.from_numpy(synth.rng(M).standard_normal((B, o.P, o.K, M, 2)).astype(np.float32))
    S = torch.view_as_complex(S) if env == "f32" else S.to(p.envelope_tensor(0).dtype)
    sums = [[O.accumulate(o, v, planes=planes) for v in values(S)] for planes in (None, [1])]
    for name in registered(p):
        y = values(p.envelopes(X))
        for b in range(B):
            assert rel(y[b], refs[b]) < STORED[env], (name, b)
        for mask, want in zip((0, 2), sums):
            A = p.accumulate(S.cuda(), plane_mask=mask).cpu().numpy().astype(np.complex128)
            for b in range(B):
                assert rel(A[b], want[b]) < 1e-6, (name, b, mask)


@pytest.mark.parametrize("env", ["bf16", "f16"])
@pytest.mark.parametrize("eps,remod,window", [(1e-3, False, "bisquare"), (1e-3, True, "bisquare"), (1e-3, True, "hann"),
                                              (0.0, True, "bisquare")])
def test_dense_storage(env, eps, remod, window):
    kw = dict(stopband_eps=eps, remodulate=remod, window=window)
    p = qtam.Plan(64.0, 8192, (3.0, 20.0), 2.0, 31.0, 5, n_out=4320, device=0, envelope=env, **kw)
    o = O.geometry(64.0, 8192, (3.0, 20.0), 2.0, 31.0, 5, n_out=4320, **kw)
    x = np.stack([synth.white(b, 8192) for b in range(3)]).astype(np.float32)
    refs = [O.forward(o, v.astype(np.float64)) for v in x]
    for name in registered(p):
        y = p.forward(torch.from_numpy(x).cuda())
        xh = p.inverse(y).cpu().double().numpy()
        for b, v in enumerate(values(y)):
            assert rel(v, refs[b]) < STORED[env], (name, b)
            assert rel(xh[b], O.inverse(o, v, tau=p.info["p_floor_rel"])) < 1e-5, (name, b)
