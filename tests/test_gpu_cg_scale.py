"""The CG solves do not depend on the units of their data: scaling y by s^2, the start value by s and alpha_0 by s^2
scales every quantity of Eq. 3 by a power of s (F is bilinear), and the gradient is linear in its cotangent.

s is a power of two, so scaling rounds nothing outside the denormal range; what may differ is the iteration at which a
solve meets its rounding floor |r| = 2^-24 |b|, by one.  One step there changes dx by at most 2^-24 |b| / alpha_n, with
alpha_n at least 1/4 of alpha_0 here: below 1e-6 of x after three Newton steps; 1e-5 leaves room for values that reach
the denormal range."""
import numpy as np
import pytest

from paper_1301_1215_gb300 import synth
from tests.helpers import ensure_built, noisy_data, rel

pytestmark = pytest.mark.gpu

NEWTON, CG = 3, 60
# |b| goes with s^3: down to 8e-9 and 2e-12 of its value, up to 6e11
SCALES = [2.0 ** -9, 2.0 ** -13, 2.0 ** 13]
SHAPES = [(16, 2), (64, 4), (64, 17), (96, 2)]       # cluster solves, four passes


def _t(a):
    import torch
    return torch.from_numpy(np.ascontiguousarray(a)).cuda()


def _problem(n, J, seed=31):
    _, fr, y = noisy_data(n, J, 11, seed=seed + n + J)
    return fr.mask, y.astype(np.complex64), synth.initial_guess(n, J).astype(np.complex64)


def _frame(n, J, s):
    from paper_1301_1215_gb300.nlinv import Nlinv
    mask, y, x0 = _problem(n, J)
    with Nlinv(n, J, newton_steps=NEWTON, cg_iters=CG, alpha0=s * s) as ctx:
        x, res = ctx.reconstruct(_t(y * np.float32(s * s)), _t(mask), _t(x0 * np.float32(s)), resid=True)
        return x.cpu().numpy() / np.float32(s), np.array(res) / (s * s), ctx.cg_stops()


def _same_stops(a, b):
    last = [CG if v < 0 else v for v in a], [CG if v < 0 else v for v in b]
    return all(abs(p - q) <= 1 for p, q in zip(*last))


@pytest.mark.parametrize("s", SCALES)
@pytest.mark.parametrize("n,J", SHAPES)
def test_scaled_frame(n, J, s):
    ensure_built()
    x1, r1, stops1 = _frame(n, J, 1.0)
    x, r, stops = _frame(n, J, s)
    assert any(v >= 0 for v in stops1)               # the floor is part of what is compared
    assert _same_stops(stops, stops1), (stops, stops1)
    assert rel(x, x1) < 1e-5
    assert np.allclose(r, r1, rtol=1e-5)


@pytest.mark.parametrize("s", SCALES)
def test_scaled_batch(s):
    ensure_built()
    from paper_1301_1215_gb300.nlinv import NlinvBatch
    shapes = [(16, 2), (64, 4), (64, 4), (96, 2)]
    problems = [_problem(n, J, 50 + i) for i, (n, J) in enumerate(shapes)]

    def run(s):
        with NlinvBatch(shapes, newton_steps=NEWTON, cg_iters=CG, alpha0=s * s) as b:
            xs, res = b.reconstruct([_t(y * np.float32(s * s)) for _, y, _ in problems], [_t(m) for m, _, _ in problems],
                                    xs=[_t(x0 * np.float32(s)) for _, _, x0 in problems], resid=True)
            return [x.cpu().numpy() / np.float32(s) for x in xs], np.array(res) / (s * s)
    x1, r1 = run(1.0)
    x, r = run(s)
    for a, b in zip(x, x1):
        assert rel(a, b) < 1e-5
    assert np.allclose(r, r1, rtol=1e-5)


@pytest.mark.parametrize("s", [2.0 ** -27, 2.0 ** -40, 2.0 ** 40])
@pytest.mark.parametrize("n,J", SHAPES)
def test_scaled_cotangent(n, J, s):
    ensure_built()
    from paper_1301_1215_gb300.nlinv import Nlinv
    mask, y, x0 = _problem(n, J)
    g = synth.random_complex((1 + J, n, n), synth.rng_for(n + J)).astype(np.complex64)
    with Nlinv(n, J, newton_steps=NEWTON, cg_iters=CG) as ctx:
        ty, tm = _t(y), _t(mask)
        _, ck = ctx.reconstruct_checkpoints(ty, tm, _t(x0))

        def run(s):
            out = ctx.reconstruct_vjp(ty, tm, ck, _t(g * np.float32(s)))
            return [v.cpu().numpy() / np.float32(s) for v in out], ctx.cg_stops()
        want, stops1 = run(1.0)
        got, stops = run(s)
    assert any(v >= 0 for v in stops1)
    assert _same_stops(stops, stops1), (stops, stops1)
    for a, b in zip(got, want):
        assert rel(a, b) < 1e-5
