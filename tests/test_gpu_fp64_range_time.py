"""FP64 flow outside the range of the integer sums costs what FP64 sums cost.

A node with a population outside [2^-6, 2^-1) sends its warp to FP64 sums, about twice the FP64
operations of the integer form.  Were each node to choose by itself, a warp with one such node
would run both forms, three times.  Step times of a state with one fast column in each warp
and of one near rest, on a lattice that fills the device (128^3, steps of 0.5 and 1.1 ms); the
limit of 2.5 lies between the two.
"""
import numpy as np
import pytest
import torch

import lbpc_inputs as inp
from paper_1703_02652_gb300 import LBPC

pytestmark = pytest.mark.gpu

E = np.array([(0, 0, 0), (1, 0, 0), (-1, 0, 0), (0, 1, 0), (0, -1, 0), (0, 0, 1), (0, 0, -1),
              (1, 1, 0), (-1, 1, 0), (1, -1, 0), (-1, -1, 0), (1, 0, 1), (-1, 0, 1), (1, 0, -1),
              (-1, 0, -1), (0, 1, 1), (0, -1, 1), (0, 1, -1), (0, -1, -1)], float)
W = np.array([1 / 3] + [1 / 18] * 6 + [1 / 36] * 12)


def _step_time(lat, f, g):
    best = np.inf
    for _ in range(6):  # the first one warms up; the fast columns live for many more steps
        lat.set_distributions(f, g)
        a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        with torch.cuda.stream(lat.stream):
            a.record()
            lat.step(3)
            b.record()
        b.synchronize()
        best = min(best, a.elapsed_time(b))
    return best


def test_one_fast_node_does_not_cost_its_warp_both_forms():
    n = 128
    p = inp.Params(precision=inp.FP64, bc=[inp.PERIODIC] * 6, Ra=1e6, Pr=0.02, St=1.0,
                   report_every=10 ** 6)
    lat = LBPC((n, n, n), p)
    g = torch.full((7, n ** 3), 1 / 16, dtype=torch.float64, device="cuda")
    g[0] += 3.0  # liquid
    x = np.arange(n ** 3) % n
    t = []
    for speed in (0.0, 0.3):
        u = np.stack([0 * x, np.where(x % 32 == 5, speed, 0.0), 0 * x])
        eu = E @ u
        f = W[:, None] * (1 + 3 * eu + 4.5 * eu ** 2 - 1.5 * (u ** 2).sum(0))
        assert ((f < 2.0 ** -6).any()) == (speed > 0)
        t.append(_step_time(lat, torch.from_numpy(f).cuda(), g))
    assert t[1] <= 2.5 * t[0], t
