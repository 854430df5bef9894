"""The CG solves of single frames against the oracle where their kernels change shape: the cluster solve (grid sides up
to 64, up to 16 coils, field of view n/4) at its smallest and largest grids and clusters, the four-pass iteration just
outside it (17 coils, another field of view, side 80) and on sides with every kind of split, with zero, one, odd and even
numbers of iterations (the solution is updated in pairs of iterations), and the gradient's solve.

Tolerance: one operator application is good to 1e-5; three Newton steps with alpha down to 1/4 amplify it by at most
about 1/alpha per solve, so 1e-4 relative on x leaves room."""
import numpy as np
import pytest

import oracle.nlinv_oracle as O
from paper_1301_1215_gb300 import synth
from tests.helpers import ensure_built, noisy_data, rel

pytestmark = pytest.mark.gpu

CASES = [(16, 1, None, 8), (16, 16, None, 7), (32, 2, None, 8), (48, 3, None, 5), (48, 16, None, 4), (64, 1, None, 6),
         (64, 16, None, 5), (64, 17, None, 5), (64, 3, 13, 6), (80, 2, None, 5), (96, 2, None, 4), (160, 2, None, 3),
         (64, 3, None, 0), (64, 3, None, 1), (64, 3, None, 2), (96, 2, None, 0), (96, 2, None, 1), (96, 2, None, 2)]


@pytest.mark.parametrize("n,J,fov,iters", CASES)
def test_solve_matches_oracle(n, J, fov, iters):
    ensure_built()
    import torch
    from paper_1301_1215_gb300.nlinv import Nlinv
    s, fr, y = noisy_data(n, J, 9, seed=900 + n + J, fov=fov)
    y64 = y.astype(np.complex64)
    x0 = synth.initial_guess(n, J)
    rng = synth.rng_for(n * 100 + J)
    # a centre that differs from the start value also off the field of view
    xref = x0 + 0.05 * synth.random_complex(x0.shape, rng) * np.concatenate(
        [np.ones((1, n, n)), np.repeat(O.sobolev_weight(n, s.a, s.l)[None], J, axis=0)])
    t = lambda a: torch.from_numpy(np.ascontiguousarray(a.astype(np.complex64))).to("cuda")
    with Nlinv(n, J, newton_steps=3, cg_iters=iters, fov=fov) as ctx:
        xg, res = ctx.reconstruct(t(y64), torch.from_numpy(fr.mask).to("cuda"), t(x0), t(xref), resid=True)
        stops = ctx.cg_stops()
    want, res_o = O.irgnm(s, fr.mask, y64.astype(np.complex128), x0.astype(np.complex64).astype(np.complex128),
                          xref.astype(np.complex64).astype(np.complex128), 3, iters)
    if iters == 0:
        assert np.array_equal(xg.cpu().numpy(), x0.astype(np.complex64))
    assert rel(xg.cpu().numpy(), want) < 1e-4, stops
    assert np.allclose(res, res_o, rtol=1e-4)


def test_cluster_and_four_pass_solves_agree_on_the_stop():
    """The same small problem with the launch shapes of the cluster solve (fov n/4) for J = 16 and of the four passes for
    J = 17 (a coil of zero data more): the floor is reached at the same iteration or one apart."""
    ensure_built()
    import torch
    from paper_1301_1215_gb300.nlinv import Nlinv
    s, fr, y = noisy_data(32, 16, 11, seed=77)
    m = torch.from_numpy(fr.mask).to("cuda")
    t = lambda a: torch.from_numpy(np.ascontiguousarray(a.astype(np.complex64))).to("cuda")
    with Nlinv(32, 16, newton_steps=2, cg_iters=30) as ctx:
        xa = ctx.reconstruct(t(y), m).cpu().numpy()
        a = ctx.cg_stops()
    y17 = np.concatenate([y, np.zeros((1, 32, 32))])
    with Nlinv(32, 17, newton_steps=2, cg_iters=30) as ctx:
        xb = ctx.reconstruct(t(y17), m).cpu().numpy()
        b = ctx.cg_stops()
    assert all(p >= 0 and q >= 0 and abs(p - q) <= 1 for p, q in zip(a, b)), (a, b)
    assert rel(xb[:17], xa) < 1e-4
    assert np.abs(xb[17]).max() < 1e-6 * np.abs(xa[1:]).max()


@pytest.mark.parametrize("n,J", [(64, 4), (96, 2)])
def test_nan_in_a_solve_is_flagged_and_leaves_nothing_behind(n, J):
    """NaN data break the first solve down (cluster solve, four passes): no step is taken, nlinv_wait says so once, and the
    next reconstruction on the context is that of a fresh one."""
    ensure_built()
    import torch
    from paper_1301_1215_gb300 import _lib
    from paper_1301_1215_gb300.nlinv import Nlinv, NlinvError
    s, fr, y = noisy_data(n, J, 11, seed=78)
    t = lambda a: torch.from_numpy(np.ascontiguousarray(a)).to("cuda")
    y = y.astype(np.complex64)
    bad = y.copy()
    bad[0, 0, 0] = np.nan                                # the centre of k-space, which every spoke samples
    x0 = synth.initial_guess(n, J).astype(np.complex64)
    with Nlinv(n, J, newton_steps=3, cg_iters=8) as ctx:
        want = ctx.reconstruct(t(y), t(fr.mask)).cpu().numpy()
    with Nlinv(n, J, newton_steps=3, cg_iters=8) as ctx:
        x = ctx.reconstruct(t(bad), t(fr.mask), t(x0)).cpu().numpy()
        assert np.array_equal(x, x0)
        assert ctx.cg_stops() == [0, 0, 0]
        with pytest.raises(NlinvError) as e:
            ctx.wait()
        assert e.value.status == _lib.EBREAKDOWN
        ctx.wait()
        assert np.array_equal(ctx.reconstruct(t(y), t(fr.mask)).cpu().numpy(), want)
