"""Calls recorded into a CUDA graph, whose kernel-to-kernel edges let each kernel start
early: replays on new inputs against the same calls made directly, at lengths that are no
power of two, in FP64, with 16-bit storage, dense tiles and a stream.

Envelopes, peaks and plane choices are the same numbers.  Accumulations add up to 40
rows a bin in whatever order they arrive: two orders differ by about 2 x sqrt(40) x 6e-8
of the partial sums, 2e-6 with those up to twice the sum (FP64: 4e-15, taken as 1e-13)."""
import pytest

from paper_2603_29785_gb300 import qtam

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

CASES = [dict(N=24576), dict(N=18000), dict(N=18000, compute="f64"), dict(N=16384, compute="f64"),
         dict(N=40960, envelope="bf16"), dict(N=12150, window="hann"),
         dict(N=1024, n_out=540, stopband_eps=1e-3, remodulate=True)]


@pytest.mark.parametrize("case", CASES, ids=lambda c: "-".join(f"{v}" for v in c.values()))
def test_replay(case):
    kw = dict(case)
    N = kw.pop("N")
    fs = N / 4.0
    p = qtam.Plan(fs, N, (6.0, 12.0), 4.0, 0.4 * fs if "stopband_eps" in kw else 60.0, 20, device=0, **kw)
    B = 3
    gen = torch.Generator(device="cuda").manual_seed(N)
    xs = [torch.randn((B, N), generator=gen, device="cuda", dtype=p.real_dtype()) for _ in range(4)]
    x = xs[0].clone()

    def calls():
        y = p.forward(x)
        return (y, p.inverse(y), p.inverse(y, plane_mask=1), *p.plane_metrics(y))

    s = torch.cuda.Stream()
    s.wait_stream(torch.cuda.current_stream())
    with torch.cuda.stream(s):
        calls()                              # the masks' tables exist before the capture
    torch.cuda.current_stream().wait_stream(s)
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g, stream=s):
        out = calls()
    tol = 1e-13 if p.compute == "f64" else 2e-6
    for v in xs[1:] + xs[:1]:
        x.copy_(v)
        for o in out[:2]:
            o.zero_()
        g.replay()
        got = [o.clone() for o in out]
        want = calls()
        assert torch.equal(got[0], want[0])
        for a, b in zip(got[1:4], want[1:4]):           # atomic sums: another order
            assert torch.linalg.norm((a - b).double()) <= tol * torch.linalg.norm(b.double())
        for a, b in zip(got[4:], want[4:]):
            assert torch.equal(a, b)


def test_replay_of_a_stream_step():
    p = qtam.Plan(2048.0, 12288, (6.0, 12.0), 8.0, 600.0, 20, n_out=768, device=0)
    a, b = (qtam.Stream(p, max_chunks=4) for _ in range(2))
    gen = torch.Generator(device="cuda").manual_seed(3)
    x = torch.randn(4 * a.hop, generator=gen, device="cuda")
    s = torch.cuda.Stream()
    for o in (a, b):
        with torch.cuda.stream(s):
            o.inverse(o.forward(x))
            o.reset()
    torch.cuda.synchronize()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g, stream=s):
        a.reset()
        y = a.forward(x)
        z = a.inverse(y)
    for seed in (5, 6):
        x.copy_(torch.randn(4 * a.hop, generator=gen.manual_seed(seed), device="cuda"))
        g.replay()
        b.reset()
        wy = b.forward(x)
        wz = b.inverse(wy)
        assert torch.equal(y, wy) and torch.linalg.norm(z - wz) <= 2e-6 * torch.linalg.norm(wz)
