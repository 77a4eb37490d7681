"""Loading and reading populations converts every double as the hardware would.

A state loaded from device arrays is rounded once to the storage precision (FP32: f - w_a and
g_a, to nearest even) and read back exactly, so the values returned are known bit for bit:
zeros of both signs, ties, the smallest and largest floats and their neighbours, values that
overflow or fall into the subnormal range, infinities and NaN.
"""
import numpy as np
import pytest
import torch

import lbpc_inputs as inp
from paper_1703_02652_gb300 import LBPC

pytestmark = pytest.mark.gpu

TINY, BIG = float(np.finfo(np.float32).tiny), float(np.finfo(np.float32).max)
SPECIAL = np.array([0.0, -0.0, 1.0, 1 + 2.0 ** -24, 1 + 3 * 2.0 ** -24, -(1 + 2.0 ** -24),
                    1 + 2.0 ** -24 + 2.0 ** -50, TINY, TINY * (1 - 2.0 ** -25), TINY / 2, 1e-45,
                    7e-46, 1e-300, 5e-324, BIG, BIG * (1 + 2.0 ** -26), BIG * (1 + 2.0 ** -24),
                    -1e300, np.inf, -np.inf, np.nan, 2.0 ** 127, 2.0 ** 128, np.pi, -1e-7])


@pytest.mark.parametrize("streaming", [inp.PULL, inp.AA])
@pytest.mark.parametrize("shape", [(25, 3, 2), (26, 1, 1)])
def test_loaded_populations_are_rounded_once_and_read_back(streaming, shape):
    N = int(np.prod(shape))
    p = inp.Params(precision=inp.FP32, streaming=streaming, bc=[inp.PERIODIC] * 6, Ra=1e5, Pr=0.7)
    w = np.array([1 / 3] + [1 / 18] * 6 + [1 / 36] * 12)
    shift = w.astype(np.float32).astype(np.float64)[:, None]
    rng = np.random.default_rng(3)
    # the special values become the stored deviations of f where w + v - w gives them back, and
    # g as they are; both among ordinary ones
    f = w[:, None] + 0.01 * rng.standard_normal((19, N))
    g = rng.uniform(0, 0.25, (7, N))
    for i, v in enumerate(SPECIAL):
        f[rng.integers(19), rng.integers(N)] = v
        f[rng.integers(19), rng.integers(N)] = v + w[0]
        g[1 + i % 6, rng.integers(N)] = v
    f[3, 0], f[0, 1] = shift[3, 0], shift[0, 0]  # stored zeros
    lat = LBPC(shape, p)
    lat.set_distributions(torch.from_numpy(f).cuda(), torch.from_numpy(g).cuda())
    f1, g1 = (v.cpu().numpy() for v in lat.distributions())
    with np.errstate(over="ignore"):
        want_f = (f - shift).astype(np.float32).astype(np.float64) + shift
        want_g = g[1:].astype(np.float32).astype(np.float64)
    assert np.array_equal(f1, want_f, equal_nan=True)
    assert np.array_equal(g1[1:], want_g, equal_nan=True)
