"""FP64 flow steps with integer sums, at the edges of the ranges they hold.

Populations in [2^-6, 2^-1) with corrections below 2^-7 and results in (0, 2^-1) take integer
sums; any other node takes FP64 sums.  One step from states on both sides of each bound, mixed
within a warp, against the oracle.  Tolerance: FP64 rounding of moments up to ~30x the
populations, 30 x 2^-53 x the largest population of the state (about 1e-13 for values of
order one).
"""
import numpy as np
import pytest
import torch

import lbpc_inputs as inp
import oracle
from paper_1703_02652_gb300 import LBPC

pytestmark = pytest.mark.gpu


def _states(shape):
    N = int(np.prod(shape))
    rng = np.random.default_rng(9)
    w = np.array([1 / 3] + [1 / 18] * 6 + [1 / 36] * 12)[:, None]
    rest = np.repeat(w, N, axis=1)
    near = rest * (1 + 0.05 * rng.uniform(-1, 1, rest.shape))
    yield "inside", near
    for name, v in (("lower bound", 2.0 ** -6), ("below", np.nextafter(2.0 ** -6, 0)),
                    ("small", 1e-9), ("zero", 0.0), ("negative", -0.01), ("upper bound", 0.5),
                    ("below the upper", np.nextafter(0.5, 0)), ("above", 0.75), ("large", 3.0)):
        f = near.copy()
        f[rng.integers(19, size=N // 5), rng.choice(N, N // 5, replace=False)] = v
        yield name, f
    # momentum whose correction passes 2^-7 in solid nodes, and results that leave (0, 1/2)
    f = near.copy()
    f[1, ::3] += 0.3
    f[2, 1::3] += 0.1
    yield "large corrections", f


@pytest.mark.parametrize("shape", [(33, 4, 3), (64, 5, 2)])
@pytest.mark.parametrize("streaming", [inp.PULL, inp.AA])
@pytest.mark.parametrize("darcy_A", [0.0, 4.0])
def test_one_step_at_the_bounds_of_the_integer_sums(shape, streaming, darcy_A):
    p = inp.Params(precision=inp.FP64, streaming=streaming, Ra=1e5, Pr=0.7, St=0.8,
                   darcy_A=darcy_A)
    _, gq = inp.random_state(shape, seed=12, flow=False)
    for name, f in _states(shape):
        g, o = LBPC(shape, p), oracle.Oracle(shape, p)
        g.set_distributions(torch.from_numpy(f).cuda(), torch.from_numpy(gq).cuda())
        f0, g0 = (v.cpu().numpy() for v in g.distributions())
        o.set_distributions(f0, g0)
        for _ in range(2):
            g.step(1)
            o.step(1)
            f1, g1 = (v.cpu().numpy() for v in g.distributions())
            fo, go = o.distributions()
            tol = 30 * 2.0 ** -53 * max(1.0, np.abs(fo).max(), np.abs(go).max()) * 10  # ten roundings
            assert np.abs(f1 - fo).max() <= tol, name
            assert np.abs(g1 - go).max() <= tol, name
            o.set_distributions(f1, g1)
