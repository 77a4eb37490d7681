"""A step of a long call takes no longer than one of a short call.

Steps are launched early: a grid becomes resident while the one before it works.  If more than one
could wait, a long call's grids would crowd the SMs, with blocks where a waiting grid left room
(12.2 us a step in calls of 1000 steps against 4.8 in calls of 50, on 16,384 nodes in FP64).  The
limit of 1.3 covers the noise of the short calls.
"""
import numpy as np
import pytest
import torch

import lbpc_inputs as inp
from paper_1703_02652_gb300 import LBPC

pytestmark = pytest.mark.gpu

I, A, P = inp.ISOTHERMAL, inp.ADIABATIC, inp.PERIODIC


@pytest.mark.parametrize("flow,precision,shape,bc", [
    (inp.FLOW_NONE, inp.FP64, (128, 1, 128), [I, I, P, P, A, A]),
    (inp.FLOW_NONE, inp.FP64, (24, 24, 24), [I, I, A, A, A, A]),
    (inp.FLOW_MRT, inp.FP32, (32, 32, 32), [I, I, A, A, A, A]),
    (inp.FLOW_NONE, inp.FP32, (40, 40, 40), [I, I, A, A, A, A])])
def test_step_time_does_not_grow_with_the_call(flow, precision, shape, bc):
    p = inp.Params(precision=precision, flow_model=flow, bc=bc, Ra=1e5, Pr=0.7,
                   tau_g=0.0 if flow else 0.9, report_every=10 ** 6)
    lat = LBPC(shape, p)
    lat.set_initial_h(np.random.default_rng(0).uniform(-0.2, 1.5, int(np.prod(shape))))
    lat.step(50)

    def us_a_step(n):
        times = []
        for _ in range(5):
            a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            torch.cuda.synchronize()
            with torch.cuda.stream(lat.stream):
                a.record()
                lat.step(n)
                b.record()
            b.synchronize()
            times.append(a.elapsed_time(b) * 1e3 / n)
        return sorted(times)[2]

    short, long = us_a_step(50), us_a_step(1000)
    assert long <= 1.3 * short, (short, long)
