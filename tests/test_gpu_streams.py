"""Operator calls on the caller's stream (nlinv_use_stream): same results as on the context's own stream, calls of one
context on several streams in order, reading the stream attribute, and capture into a CUDA graph."""
import numpy as np
import pytest

from tests.helpers import ensure_built
from paper_1301_1215_gb300 import synth

pytestmark = pytest.mark.gpu

N, J = 64, 3


@pytest.fixture(scope="module")
def env():
    ensure_built()
    import torch
    dev = torch.device("cuda")
    rng = synth.rng_for(4242)
    t = lambda a: torch.from_numpy(np.ascontiguousarray(a.astype(np.complex64))).to(dev)
    xs = [t(synth.random_complex((1 + J, N, N), rng)) for _ in range(4)]
    mask = torch.from_numpy(synth.radial_mask(N, 9)).to(dev)
    return torch, xs, mask


def _on_own_stream(torch, xs, mask):
    from paper_1301_1215_gb300.nlinv import Nlinv
    with Nlinv(N, J) as ctx:
        ctx.stream                           # every later call runs on the context's stream
        out = [ctx.forward(x, mask) for x in xs]
        adj = [ctx.adjoint(xs[0], mask, y) for y in out]
    torch.cuda.synchronize()
    return out, adj


def test_calls_on_several_streams_keep_their_order(env):
    torch, xs, mask = env
    from paper_1301_1215_gb300.nlinv import Nlinv
    want_f, want_a = _on_own_stream(torch, xs, mask)
    streams = [torch.cuda.Stream() for _ in range(3)]
    torch.cuda.synchronize()
    with Nlinv(N, J) as ctx:
        got_f, got_a = [], []
        for i, x in enumerate(xs):           # one workspace, a stream per call, nothing waited for in between
            with torch.cuda.stream(streams[i % 3]):
                y = ctx.forward(x, mask)
                got_f.append(y)
                got_a.append(ctx.adjoint(xs[0], mask, y))
        rec = ctx.reconstruct(want_f[0], mask)          # the context's own stream, after the calls above
        torch.cuda.synchronize()
        for g, w in zip(got_f + got_a, want_f + want_a):
            assert torch.equal(g, w)
    with Nlinv(N, J) as ctx:
        assert torch.equal(rec, ctx.reconstruct(want_f[0], mask))


def test_reading_the_stream_orders_it_after_the_calls(env):
    torch, xs, mask = env
    from paper_1301_1215_gb300.nlinv import Nlinv
    want_f, _ = _on_own_stream(torch, xs, mask)
    with Nlinv(N, J) as ctx:
        y = ctx.forward(xs[1], mask)
        s = ctx.stream
        with torch.cuda.stream(s):
            z = y * 1.0                      # on the context's stream, without another wait
        s.synchronize()
        assert torch.equal(z, want_f[1])
        y2 = ctx.forward(xs[2], mask)        # now on the context's stream, the current stream waits for it
        assert torch.equal(y2, want_f[2])


def test_a_refused_call_uses_up_the_choice(env):
    torch, xs, mask = env
    import ctypes as C
    from paper_1301_1215_gb300.nlinv import Nlinv
    side = torch.cuda.Stream()
    with Nlinv(N, J) as ctx:
        lib, h = ctx._lib, ctx._h
        assert lib.nlinv_use_stream(h, C.c_void_p(side.cuda_stream)) == 1
        assert lib.nlinv_forward(h, None, None, None) != 0
        assert lib.nlinv_use_stream(h, C.c_void_p(ctx._stream.cuda_stream)) == 0
        assert lib.nlinv_use_stream(None, None) == 0


def test_captured_calls_replay(env):
    torch, xs, mask = env
    from paper_1301_1215_gb300.nlinv import Gridder, Nlinv
    want_f, want_a = _on_own_stream(torch, xs, mask)
    ang = [(np.cos(a), np.sin(a)) for a in (0.1, 1.2, 2.3)]
    smp = torch.randn((J, 3, 2 * N), dtype=torch.complex64, device="cuda")
    with Nlinv(N, J) as ctx, Gridder(N, ang) as gr:
        ctx.forward(xs[3], mask)             # a call outside the capture, on the default stream
        yg, mg = gr.grid(smp)
        x = xs[0].clone()
        torch.cuda.synchronize()
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g):
            y = ctx.forward(x, mask)
            a = ctx.adjoint(xs[0], mask, y)
            yc, mc = gr.grid(smp)
        for k in (1, 2):
            x.copy_(xs[k])
            g.replay()
            torch.cuda.synchronize()
            assert torch.equal(y, want_f[k]) and torch.equal(a, want_a[k])
        assert torch.equal(yc, yg) and torch.equal(mc, mg)
        assert torch.equal(ctx.forward(xs[3], mask), want_f[3])      # and calls outside the capture go on
