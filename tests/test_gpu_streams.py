"""One plan on several streams and threads at once: every call has the scratch, the
tables and the order of kernels it needs, whatever runs beside it."""
import threading

import pytest

from paper_2603_29785_gb300 import qtam

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

ARGS = (4096.0, 65536, (8.0, 16.0), 20.0, 1024.0, 24)


def inputs(p, n, B=6):
    gen = torch.Generator(device="cuda").manual_seed(n)
    return [torch.randn((B, p.N), generator=gen, device="cuda", dtype=p.real_dtype()) for _ in range(n)]


def same(a, b, tol=1e-6):
    # the inverse sums with atomics: FP32 rounding of another order, 6e-8 sqrt(terms) < 1e-6
    return float(torch.linalg.norm(a - b) / torch.linalg.norm(b)) < tol


@pytest.mark.parametrize("explicit", [True, False])
def test_two_streams(explicit):
    p = qtam.Plan(*ARGS, device=0)
    xs = inputs(p, 2)
    want = [(y := p.forward(x), p.inverse(y)) for x in xs]
    streams = [torch.cuda.Stream() for _ in xs]
    torch.cuda.synchronize()
    assert len({p.workspace(6, s)[0].data_ptr() for s in (*streams, None)}) == 3
    out = [[] for _ in xs]
    for _ in range(20):
        for i, s in enumerate(streams):
            if explicit:
                y = p.forward(xs[i], stream=s)
                out[i].append((y, p.inverse(y, stream=s)))
            else:
                with torch.cuda.stream(s):
                    y = p.forward(xs[i])
                    out[i].append((y, p.inverse(y)))
    torch.cuda.synchronize()
    for i, (wy, wx) in enumerate(want):
        for y, x in out[i]:
            assert torch.equal(y, wy) and same(x, wx)


def test_two_threads_on_one_stream():
    p = qtam.Plan(*ARGS, device=0)
    xs = inputs(p, 2)
    want = [(y := p.forward(x), p.inverse(y)) for x in xs]
    bad = []

    def work(i):
        for _ in range(30):
            y = p.forward(xs[i])
            x = p.inverse(y)
            if not (torch.equal(y, want[i][0]) and same(x, want[i][1])):
                bad.append(i)

    ts = [threading.Thread(target=work, args=(i,)) for i in range(2)]
    [t.start() for t in ts]
    [t.join() for t in ts]
    assert not bad


@pytest.mark.parametrize("compute", ["f32", "f64"])
def test_new_tables_on_a_non_blocking_stream(compute):
    """The first launch that reads a new plan's, mask's or stream's tables, on a stream
    that does not wait for the legacy one, against a plan whose tables are long there."""
    old = qtam.Plan(*ARGS, compute=compute, device=0)
    x = inputs(old, 1)[0]
    wy = old.forward(x)
    wx = old.inverse(wy, plane_mask=2)
    torch.cuda.synchronize()
    tol = 1e-13 if compute == "f64" else 1e-6
    for _ in range(5):
        s = torch.cuda.Stream()
        with torch.cuda.stream(s):
            p = qtam.Plan(*ARGS, compute=compute, device=0)
            y = p.forward(x)
            xh = p.inverse(y, plane_mask=2)
            st = qtam.Stream(p, max_chunks=2)
            z = st.forward(x[0, :st.hop].clone())
        s.synchronize()
        assert torch.equal(y, wy) and same(xh, wx, tol)
        st0 = qtam.Stream(old, max_chunks=2)
        assert torch.equal(z, st0.forward(x[0, :st0.hop].clone()))


def test_outputs_belong_to_the_stream_that_writes_them():
    """A block freed on the current stream, whose kernels may not have run, is not handed to a call on
    another stream; an output read on the current stream is not reused by its own before that has run."""
    p = qtam.Plan(*ARGS, device=0)
    x = inputs(p, 1)[0]
    s = torch.cuda.Stream()
    want = p.forward(x)
    p.forward(x, stream=s)
    torch.cuda.synchronize()
    old = p.envelope_tensor(6)
    at = old.data_ptr()
    del old
    y = p.forward(x, stream=s)
    assert y.data_ptr() != at
    del y
    outs = [p.forward(x, stream=s), p.inverse(want, stream=s), p.spectrum(x, stream=s), *p.plane_metrics(want, stream=s)]
    s.synchronize()
    assert torch.equal(outs[0], want) and same(outs[1], p.inverse(want)) and torch.equal(outs[2], p.spectrum(x))
    assert all(torch.equal(a, b) for a, b in zip(outs[4:], p.plane_metrics(want)[1:]))
    at = outs[0].data_ptr()
    torch.cuda._sleep(20_000_000)                    # the current stream is busy about 10 ms
    twice = outs[0] + outs[0]
    del outs
    y = p.forward(x, stream=s)
    assert y.data_ptr() != at
    torch.cuda.synchronize()
    assert torch.equal(twice, want + want)


def test_replay_after_the_capturing_thread_has_ended():
    """The scratch a captured call recorded is not given to anyone else while the plan lives."""
    p = qtam.Plan(*ARGS, device=0)
    x, other = inputs(p, 2)
    want = p.forward(x)
    made = {}

    def capture():
        s = torch.cuda.Stream()
        with torch.cuda.stream(s):
            p.forward(other)                              # this thread's scratch on s, before the capture
        s.synchronize()
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g, stream=s):
            made["y"] = p.forward(x)
        made.update(g=g, s=s, ws=p.workspace(6, s)[0].data_ptr())

    t = threading.Thread(target=capture)
    t.start()
    t.join()
    with torch.cuda.stream(made["s"]):                    # new blocks of that stream's pool are others
        taken = [torch.empty(p.workspace(6, 0)[1], dtype=torch.uint8, device="cuda") for _ in range(4)]
    assert made["ws"] not in [b.data_ptr() for b in taken]
    made["g"].replay()
    assert torch.equal(made["y"], want)
