"""Calls of one context or gridder that follow one another over streams while the first stream is still busy: a finite
delay on the first stream keeps its call from starting, so that a call on the second that did not wait would change the
workspace under it (or run ahead of it)."""
import ctypes as C

import numpy as np
import pytest

from paper_1301_1215_gb300 import synth
from tests.helpers import ensure_built

pytestmark = pytest.mark.gpu

N, J = 64, 3
DELAY = 20_000_000            # clock cycles of one spinning thread: about 10 ms, against some 30 us of a call


@pytest.fixture(scope="module")
def env():
    ensure_built()
    import torch
    rng = synth.rng_for(515)
    t = lambda a: torch.from_numpy(np.ascontiguousarray(a)).cuda()
    xs = [t(synth.random_complex((1 + J, N, N), rng).astype(np.complex64)) for _ in range(2)]
    mask = t(synth.radial_mask(N, 9))
    from paper_1301_1215_gb300.nlinv import Nlinv
    with Nlinv(N, J) as ctx:
        want = [ctx.forward(x, mask).cpu() for x in xs]
    return torch, xs, mask, want


def test_second_stream_follows_a_busy_first(env):
    torch, xs, mask, want = env
    from paper_1301_1215_gb300.nlinv import Nlinv
    s = [torch.cuda.Stream() for _ in range(2)]
    out = [torch.empty((J, N, N), dtype=torch.complex64, device="cuda") for _ in range(2)]
    with Nlinv(N, J) as ctx:
        ctx.forward(xs[0], mask)
        torch.cuda.synchronize()
        for i in range(2):
            with torch.cuda.stream(s[i]):
                if i == 0:
                    torch.cuda._sleep(DELAY)
                ctx.forward(xs[i], mask, out=out[i])
        assert not s[1].query()                    # it waits behind the delay
        rec = ctx.stream                           # and so does the context's own stream
        assert not rec.query()
        torch.cuda.synchronize()
    for o, w in zip(out, want):
        assert torch.equal(o.cpu(), w)


def test_a_new_stream_at_a_destroyed_ones_handle_follows_its_call(env):
    torch, xs, mask, want = env
    from paper_1301_1215_gb300.nlinv import Nlinv
    rt = torch.cuda.cudart()
    out = [torch.empty((J, N, N), dtype=torch.complex64, device="cuda") for _ in range(2)]
    with Nlinv(N, J) as ctx:
        lib = ctx._lib

        def forward_on(handle, i):
            assert lib.nlinv_use_stream(ctx._h, C.c_void_p(handle)) == 1
            assert lib.nlinv_forward(ctx._h, xs[i].data_ptr(), mask.data_ptr(), out[i].data_ptr()) == 0
        torch.cuda.synchronize()
        first = C.c_void_p()
        assert int(rt.cudaStreamCreate(C.addressof(first))) == 0
        with torch.cuda.stream(torch.cuda.ExternalStream(first.value)):
            torch.cuda._sleep(DELAY)
        forward_on(first.value, 0)
        assert int(rt.cudaStreamDestroy(first.value)) == 0      # its work goes on
        later = [C.c_void_p() for _ in range(4)]
        for h in later:
            assert int(rt.cudaStreamCreate(C.addressof(h))) == 0
        handle = next((h.value for h in later if h.value == first.value), later[0].value)
        forward_on(handle, 1)
        ctx.wait()
        torch.cuda.synchronize()
        for h in later:
            assert int(rt.cudaStreamDestroy(h.value)) == 0
    for o, w in zip(out, want):
        assert torch.equal(o.cpu(), w)


def test_per_thread_stream(env):
    torch, xs, mask, want = env
    import threading
    from paper_1301_1215_gb300.nlinv import Nlinv
    out = [torch.empty((J, N, N), dtype=torch.complex64, device="cuda") for _ in range(2)]
    status = []
    with Nlinv(N, J) as ctx:
        lib = ctx._lib
        torch.cuda.synchronize()

        def work(i):                       # cudaStreamPerThread: handle 2, a stream of each host thread
            torch.cuda.set_device(ctx.device)
            if i == 0:
                with torch.cuda.stream(torch.cuda.ExternalStream(2)):
                    torch.cuda._sleep(DELAY)
            status.append(lib.nlinv_use_stream(ctx._h, C.c_void_p(2)))
            status.append(lib.nlinv_forward(ctx._h, xs[i].data_ptr(), mask.data_ptr(), out[i].data_ptr()))
        for i in range(2):
            th = threading.Thread(target=work, args=(i,))
            th.start()
            th.join()
        ctx.wait()
        torch.cuda.synchronize()
    assert status == [1, 0, 1, 0]
    for o, w in zip(out, want):
        assert torch.equal(o.cpu(), w)


def _spokes(k=4):
    return [(np.cos(a), np.sin(a)) for a in np.arange(k) * 0.7]


def test_gridder_shared_by_two_threads(env):
    """Each thread grids samples that its own stream produces after a delay, again and again, on one gridder."""
    torch = env[0]
    import threading
    from paper_1301_1215_gb300.nlinv import Gridder
    base = torch.randn((J, 4, 2 * N), dtype=torch.complex64, device="cuda")
    with Gridder(N, _spokes()) as gr:
        want = gr.grid(base)[0] * 2.0           # powers of two below: exact
        torch.cuda.synchronize()
        got, errors = [[], []], []

        def work(i):
            try:
                s = torch.cuda.Stream()
                with torch.cuda.stream(s):
                    for k in range(40):
                        if k % 10 == 0:
                            torch.cuda._sleep(DELAY // 10)
                        got[i].append(gr.grid(base * 2.0)[0])
                s.synchronize()
            except Exception as e:              # reported by the main thread
                errors.append(e)
        threads = [threading.Thread(target=work, args=(i,)) for i in range(2)]
        for t in threads:
            t.start()
        for t in threads:
            t.join()
        assert not errors, errors
        torch.cuda.synchronize()
        for y in got[0] + got[1]:
            assert torch.equal(y, want)


def test_gridders_stream_follows_calls_on_other_streams(env):
    torch = env[0]
    from paper_1301_1215_gb300.nlinv import Gridder
    smp = torch.randn((J, 4, 2 * N), dtype=torch.complex64, device="cuda")
    side = torch.cuda.Stream()
    with Gridder(N, _spokes()) as gr:
        gr.grid(smp)
        torch.cuda.synchronize()
        with torch.cuda.stream(side):
            torch.cuda._sleep(DELAY)
            gr.grid(smp)
        own = gr.stream                          # read with the default stream current, which has nothing to wait for
        assert not own.query()
        own.synchronize()
        assert side.query()


def test_the_stream_of_a_closed_context_can_still_be_read(env):
    torch, xs, mask, want = env
    from paper_1301_1215_gb300.nlinv import Gridder, Nlinv
    with Nlinv(N, J) as ctx, Gridder(N, _spokes()) as gr:
        y = ctx.forward(xs[0], mask)
    ctx.stream.synchronize()
    gr.stream.synchronize()
    assert torch.equal(y.cpu(), want[0])
