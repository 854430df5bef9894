"""Arrays that do not start on a 16-byte boundary (slices of larger tensors): every call gives the bits that it gives for
the same values on one, although its passes copy planes into shared memory in 16-byte pieces."""
import ctypes as C

import numpy as np
import pytest

from paper_1301_1215_gb300 import synth
from tests.helpers import ensure_built

pytestmark = pytest.mark.gpu


def _off(t, elements):
    """The values of t in memory that starts `elements` entries after a boundary."""
    import torch
    buf = torch.empty(t.numel() + elements, dtype=t.dtype, device=t.device)
    out = buf[elements:].view(t.shape)
    out.copy_(t)
    assert out.data_ptr() % 16 != 0 and out.is_contiguous()
    return out


def _inputs(n, J):
    import torch
    ensure_built()
    rng = synth.rng_for(n + 3 * J)
    t = lambda a: torch.from_numpy(np.ascontiguousarray(a)).cuda()
    x, d, r = (t(synth.random_complex((k, n, n), rng).astype(np.complex64)) for k in (1 + J, 1 + J, J))
    return x, d, r, t(synth.radial_mask(n, 9))


@pytest.mark.parametrize("n,J,fov,tensor_dft", [(16, 1, 8, False), (64, 3, 16, False), (48, 2, 11, False),
                                                (128, 2, 32, False), (256, 1, 64, True)])
@pytest.mark.parametrize("mask_off", [1, 8])
def test_operators(n, J, fov, tensor_dft, mask_off):
    from paper_1301_1215_gb300.nlinv import Nlinv
    x, d, r, m = _inputs(n, J)
    xo, do, ro, mo = _off(x, 1), _off(d, 1), _off(r, 1), _off(m, mask_off)
    with Nlinv(n, J, fov=fov, newton_steps=2, cg_iters=3, tensor_dft=tensor_dft) as ctx:
        calls = [lambda x, d, r, m, o: ctx.forward(x, m, out=o), lambda x, d, r, m, o: ctx.derivative(x, m, d, out=o),
                 lambda x, d, r, m, o: ctx.simulate(x[0], r, m, out=o),
                 lambda x, d, r, m, o: ctx.adjoint(x, m, r, out=o), lambda x, d, r, m, o: ctx.normal(x, m, d, 0.25, out=o)]
        first = ctx.reconstruct(r, m)
        for k, call in enumerate(calls):
            out = _off(r if k < 3 else x, 1)
            want = call(x, d, r, m, None)
            assert np.array_equal(call(xo, do, ro, mo, out).cpu().numpy(), want.cpu().numpy()), k
        assert np.array_equal(ctx.image(xo).cpu().numpy(), ctx.image(x).cpu().numpy())
        assert np.array_equal(ctx.reconstruct(ro, mo).cpu().numpy(), first.cpu().numpy())


def test_gradient_through_a_reconstruction():
    import torch
    from paper_1301_1215_gb300 import _lib
    from paper_1301_1215_gb300.nlinv import Nlinv
    n, J, steps = 64, 3, 2
    x, g, y, m = _inputs(n, J)
    with Nlinv(n, J, newton_steps=steps, cg_iters=5) as ctx:
        _, ck = ctx.reconstruct_checkpoints(y, m)
        want = ctx.reconstruct_vjp(y, m, ck, g)
        ins = [_off(y, 1), _off(m, 1), _off(ck, 1), _off(g, 1)]
        outs = [_off(w, 1) for w in want]
        torch.cuda.synchronize()
        p = lambda t: C.c_void_p(t.data_ptr())
        _lib.check(ctx._lib.nlinv_reconstruct_vjp(ctx._h, *map(p, ins), 0, *map(p, outs)), ctx._h)
        ctx.wait()
        for a, b in zip(outs, want):
            assert np.array_equal(a.cpu().numpy(), b.cpu().numpy())
        xs, cks = ctx.reconstruct_checkpoints(_off(y, 1), _off(m, 3), _off(x, 1))
        x1, ck1 = ctx.reconstruct_checkpoints(y, m, x)
        assert np.array_equal(cks.cpu().numpy(), ck1.cpu().numpy()) and np.array_equal(xs.cpu().numpy(), x1.cpu().numpy())


def test_forward_without_a_context():
    import torch
    from paper_1301_1215_gb300 import _lib
    n, J = 64, 3
    x, _, y, m = _inputs(n, J)
    lib = _lib.load()
    prm = _lib.Params()
    lib.nlinv_default_params(C.byref(prm), n, J)
    p = lambda t: C.c_void_p(t.data_ptr())
    got = []
    for a, b in ((x, m), (_off(x, 1), _off(m, 1))):
        out = torch.empty_like(y)
        torch.cuda.synchronize()
        _lib.check(lib.nlinv_forward_noalloc(C.byref(prm), None, p(a), p(b), p(out)))
        torch.cuda.synchronize()
        got.append(out.cpu().numpy())
    assert np.array_equal(got[0], got[1])
