"""Which kernels a step call runs on small lattices, and that they agree.

Lattices of up to 8192 nodes (3584 in FP64) take four or more steps of a call in one launch; with
fewer, with flow in other storage than FP32 and with the drag closure every step is a launch of its
own.  The launch counts tell the two apart.  The first half holds blocks to single steps bit for
bit, the second runs the single-step kernels (node pairs above all) at small shapes against the
oracle, in calls of at most three steps.
"""
import numpy as np
import pytest
import torch

import lbpc_inputs as inp
import oracle
from paper_1703_02652_gb300 import LBPC

pytestmark = pytest.mark.gpu

I, A, P = inp.ISOTHERMAL, inp.ADIABATIC, inp.PERIODIC
KEYS = ("T", "fl", "h", "rho", "u")


def _launches(lat, n):
    before = lat.launch_count
    lat.step(n)
    return lat.launch_count - before


def _by_threes(lat, n):
    """n steps, each a launch of its own."""
    count = sum(_launches(lat, min(3, n - i)) for i in range(0, n, 3))
    assert count >= n
    return lat


def _params(flow, precision, streaming, **kw):
    kw.setdefault("tau_g", 0.0 if flow or "lambda_s" in kw else 0.9)
    return inp.Params(flow_model=flow, precision=precision, streaming=streaming, Ra=1e5, Pr=0.7,
                      T_wall=[1.0, 0.1, 0.3, 0.8, 0.6, 0.2], **kw)


@pytest.mark.parametrize("flow,precision,largest,above", [
    (inp.FLOW_MRT, inp.FP32, (64, 8, 16), (64, 8, 17)),
    (inp.FLOW_SRT, inp.FP32, (8192, 1, 1), (8194, 1, 1)),
    (inp.FLOW_NONE, inp.FP64, (16, 16, 14), (17, 16, 14)),
    (inp.FLOW_NONE, inp.FP32, (128, 1, 64), (129, 1, 64)),
    (inp.FLOW_NONE, inp.FP16, (64, 8, 16), (64, 8, 17)),
    (inp.FLOW_NONE, inp.BF16, (64, 8, 16), (64, 8, 17)),
    (inp.FLOW_NONE, inp.FP16_G32, (64, 8, 16), (64, 8, 17)),
    (inp.FLOW_NONE, inp.BF16_G32, (64, 8, 16), (64, 8, 17))])
@pytest.mark.parametrize("streaming", [inp.PULL, inp.AA])
def test_small_lattices_step_in_blocks(flow, precision, largest, above, streaming):
    p = _params(flow, precision, streaming, report_every=1000)
    a = LBPC(largest, p)
    assert _launches(a, 23) == 1
    assert _launches(a, 4) == 1
    assert _launches(a, 3) == 3
    assert _launches(LBPC(above, p), 23) == 23


@pytest.mark.parametrize("flow,precision,kw", [
    (inp.FLOW_MRT, inp.FP64, {}), (inp.FLOW_MRT, inp.FP16, {}), (inp.FLOW_MRT, inp.BF16_G32, {}),
    (inp.FLOW_MRT, inp.FP32, dict(darcy_A=4.0))])
def test_other_lattices_step_one_by_one(flow, precision, kw):
    assert _launches(LBPC((8, 8, 8), _params(flow, precision, inp.PULL, report_every=1000, **kw)), 23) == 23


def _equal(a, b):
    for x, y in zip(a.distributions(), b.distributions()):
        assert (x is None and y is None) or torch.equal(x, y)
    for k, v in a.fields().items():
        assert torch.equal(v, b.fields()[k]), k


@pytest.mark.parametrize("precision", [inp.FP64, inp.FP32, inp.FP16, inp.BF16, inp.FP16_G32])
@pytest.mark.parametrize("streaming", [inp.PULL, inp.AA])
@pytest.mark.parametrize("enth_model,kw", [
    (inp.ENTH_MRT, dict(lambda_s=1.0, lambda_l=0.25, Cp_l=2.0)),
    (inp.ENTH_MRT, dict(lambda_s=0.3, lambda_l=0.5, sigma4=1.1)),
    (inp.ENTH_SRT, dict(lambda_s=0.2, lambda_l=0.4)), (inp.ENTH_SRT, {}),
    (inp.ENTH_MRT, dict(Cp_s=0.7, Cp_l=1.3, sigma4=1.9))])
def test_blocks_of_conduction_steps_equal_single_steps(precision, streaming, enth_model, kw):
    for shape, bc in (((31, 5, 6), [I, A, A, I, I, A]), ((40, 1, 12), [I, I, P, P, A, A])):
        p = _params(inp.FLOW_NONE, precision, streaming, enth_model=enth_model, bc=bc, **kw)
        h0 = np.random.default_rng(4).uniform(-0.3, 1.8, int(np.prod(shape)))
        a, b = LBPC(shape, p), LBPC(shape, p)
        for v in (a, b):
            v.set_initial_h(h0)
        for n in (23, 8):  # the second block starts at an odd step
            assert _launches(a, n) < n
            _by_threes(b, n)
            _equal(a, b)


@pytest.mark.parametrize("flow_model", [inp.FLOW_MRT, inp.FLOW_SRT])
@pytest.mark.parametrize("streaming", [inp.PULL, inp.AA])
def test_blocks_of_flow_steps_equal_single_steps(flow_model, streaming):
    for shape, bc in (((33, 9, 6), [I, A, A, I, I, A]), ((40, 1, 30), [I, I, P, P, A, A]),
                      ((16, 16, 16), [P, P, I, A, P, P])):
        p = _params(flow_model, inp.FP32, streaming, bc=bc, Cp_l=1.4)
        h0 = np.random.default_rng(5).uniform(-0.3, 1.8, int(np.prod(shape)))
        a, b = LBPC(shape, p), LBPC(shape, p)
        for v in (a, b):
            v.set_initial_h(h0)
        for n in (51, 12):
            assert _launches(a, n) < n
            _by_threes(b, n)
            _equal(a, b)


@pytest.mark.parametrize("flow,precision", [(inp.FLOW_MRT, inp.FP32), (inp.FLOW_NONE, inp.FP64)])
@pytest.mark.parametrize("streaming", [inp.PULL, inp.AA])
def test_calls_longer_than_a_block(flow, precision, streaming):
    """A launch holds 2048 steps at most; the next one goes on from there."""
    p = _params(flow, precision, streaming, report_every=10 ** 6)
    a, b = LBPC((6, 4, 5), p), LBPC((6, 4, 5), p)
    assert _launches(a, 4101) == 3  # 2048, 2048 and 5
    _by_threes(b, 4101)
    _equal(a, b)


# ---- the single-step kernels at the shapes of test_gpu_parity.py (tolerances from there) ----
def _oracle(shape, p, h0, n):
    o = oracle.Oracle(shape, p)
    o.set_initial_h(h0)
    o.step(n)
    return o


@pytest.mark.parametrize("streaming", [inp.PULL, inp.AA])
@pytest.mark.parametrize("shape,n", [((512, 4, 3), 300), ((24, 16, 12), 400), ((16, 9, 7), 40)])
def test_single_steps_of_fp32_pairs_track_oracle(shape, n, streaming):
    p = inp.Params(precision=inp.FP32, streaming=streaming, Ra=1e5, Pr=0.71, St=1.0)
    h0 = np.random.default_rng(7).uniform(-1e-6, 1e-6, int(np.prod(shape)))
    g = LBPC(shape, p)
    g.set_initial_h(h0)
    F = {k: v.cpu().numpy() for k, v in _by_threes(g, n).fields().items()}
    o = _oracle(shape, p, h0, n)
    R = o.fields()
    for k in ("T", "fl", "rho", "h"):
        assert np.abs(F[k] - R[k]).max() <= 1e-5, k
    sg = g.scalars()
    assert abs(sg["sum_h"] - F["h"].sum()) <= 1e-12 * abs(F["h"]).sum()
    assert abs(sg["sum_h"] - o.diagnostics()["sum_h"]) <= 1e-5 * F["h"].size


def test_single_steps_of_fp32_aa_and_pull_agree():
    shape, res = (16, 12, 10), {}
    for streaming in (inp.PULL, inp.AA):
        g = LBPC(shape, inp.Params(precision=inp.FP32, streaming=streaming, Ra=5e4, Pr=0.7, St=1.0))
        g.set_initial_h(np.linspace(-0.2, 1.5, int(np.prod(shape))))
        res[streaming] = _by_threes(g, 41).fields()
    for k in KEYS:
        assert (res[inp.PULL][k] - res[inp.AA][k]).abs().max() <= 2e-6, k


@pytest.mark.parametrize("streaming", [inp.PULL, inp.AA])
def test_single_steps_continue_from_a_saved_state(streaming):
    shape = (12, 10, 8)
    p = inp.Params(precision=inp.FP32, streaming=streaming, Ra=5e4, Pr=0.7, St=1.0)
    g = LBPC(shape, p)
    g.set_initial_h(np.zeros(int(np.prod(shape))))
    blob = _by_threes(g, 11).save()
    g2 = LBPC(shape, p)
    g2.load(blob)
    assert g2.step_count == 11
    _equal(_by_threes(g, 9), _by_threes(g2, 9))
