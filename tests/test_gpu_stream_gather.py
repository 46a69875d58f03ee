"""Chunk assembly of a stream: 16-byte and single-sample copies give the same chunks,
also for hops that are no multiple of four, and a reset stream is a new one."""
import pytest

from paper_2603_29785_gb300 import qtam

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("compute", ["f32", "f64"])
@pytest.mark.parametrize("N,n_out,hop", [(1024, 128, 512), (1024, 128, 16), (1000, 1000, 502), (1000, 500, 1000),
                                         (4500, 300, 4470)])
def test_chunks_and_reset(compute, N, n_out, hop):
    fs = N / 4.0
    p = qtam.Plan(fs, N, (8.0, 16.0), 8.0, 0.3 * fs, 6, max_window_hz=15.0, n_out=n_out, compute=compute, device=0)
    s = qtam.Stream(p, hop=hop, max_chunks=3)
    J = 7
    gen = torch.Generator(device="cuda").manual_seed(N + hop)
    big = torch.randn(J * hop + 1, generator=gen, device="cuda", dtype=p.real_dtype())
    x = big[1:]                                        # not 16-byte aligned
    a = s.forward(x)
    xa = s.inverse(a)
    # the definition: chunk i starts at i hop - 2 G, its central columns kept, referred to the stream's origin
    cat = torch.cat([x.new_zeros(2 * s.guard), x])
    chunks = torch.stack([cat[i * hop:i * hop + N] for i in range(J)])
    env = p.forward(chunks)
    kc = torch.from_numpy(p.geometry.kc).cuda()
    tol = 1e-12 if compute == "f64" else 1e-6
    for i in range(J):
        t = ((kc * (i * hop - 2 * s.guard)) % N).double() * (-2 * torch.pi / N)
        g = s.info["guard_cols"]
        want = env[i, :, :, g:g + s.hop_cols].to(torch.complex128) * torch.polar(torch.ones_like(t), t)[..., None]
        got = a[:, :, i * s.hop_cols:(i + 1) * s.hop_cols].to(torch.complex128)
        assert torch.linalg.norm(got - want) <= tol * torch.linalg.norm(want), i
    for push in (1, 2):                                # histories of both buffers hold samples, then a reset
        s.forward(x[:push * hop].clone())
        s.inverse(a[:, :, :push * s.hop_cols].contiguous())
        s.reset()
        b = s.forward(x.clone())                       # aligned
        assert torch.equal(a, b)
        xb = s.inverse(b)
        assert torch.linalg.norm(xb - xa) <= tol * torch.linalg.norm(xa)   # atomic sums: another order
        s.reset()
