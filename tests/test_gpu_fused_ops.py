"""The operators' fused passes (coil maps formed in the pass that uses them, two arrays in one row launch) where the two
arrays' rows share a block: odd numbers of rows per block, one coil, the most coils, ragged fields of view, and between
reconstructions, whose residual buffer they use.

Tolerance: 1e-5 relative, the bar of a single operator application in FP32."""
import numpy as np
import pytest

import oracle.nlinv_oracle as O
from paper_1301_1215_gb300 import synth
from tests.helpers import ensure_built, noisy_data, rel

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,J,fov", [(16, 1, 8), (16, 63, 3), (48, 7, 11), (96, 1, 24), (80, 5, 19),
                                     (160, 3, 40), (320, 2, 79)])
def test_operators_between_reconstructions(n, J, fov):
    ensure_built()
    import torch
    from paper_1301_1215_gb300.nlinv import Nlinv
    s, fr, y = noisy_data(n, J, 9, seed=60 + n + J, fov=fov)
    rng = synth.rng_for(n + J)
    c64 = lambda a: a.astype(np.complex64)
    x, d, r = (c64(synth.random_complex((k, n, n), rng)) for k in (1 + J, 1 + J, J))
    t = lambda a: torch.from_numpy(np.ascontiguousarray(a)).to("cuda")
    m = t(fr.mask)
    x128, d128, r128 = (a.astype(np.complex128) for a in (x, d, r))
    c = O.coils(s, x128)
    with Nlinv(n, J, newton_steps=2, cg_iters=3, fov=fov) as ctx:
        first = ctx.reconstruct(t(c64(y)), m)
        assert rel(ctx.forward(t(x), m).cpu().numpy(), O.forward(s, fr.mask, x128)) < 1e-5
        assert rel(ctx.derivative(t(x), m, t(d)).cpu().numpy(), O.derivative(s, fr.mask, x128, d128, c)) < 1e-5
        assert rel(ctx.adjoint(t(x), m, t(r)).cpu().numpy(), O.adjoint(s, fr.mask, x128, r128, c)) < 1e-5
        assert rel(ctx.normal(t(x), m, t(d), 0.125).cpu().numpy(), O.normal(s, fr.mask, x128, d128, 0.125, c)) < 1e-5
        assert torch.equal(ctx.reconstruct(t(c64(y)), m), first)
