"""The step kernels at the lattice shapes where their launches change.

* Rows that fill whole blocks, rows counted in memory order within each z plane, and
  lattices counted in one run, each at its edges: one step from a random state against the
  oracle, with walls and wall temperatures on every face (tolerances of
  test_gpu_parity.py: FP32 moments up to ~30x the populations, 5e-6; FP16 one ulp of a
  stored deviation, 2.5e-4, six of them on the rest channel).
* Blocks of steps in one launch (small lattices): the same bits as the steps one by one,
  since both run the same arithmetic on the same stored values.
"""
import numpy as np
import pytest
import torch

import lbpc_inputs as inp
import oracle
from paper_1703_02652_gb300 import LBPC

pytestmark = pytest.mark.gpu

I, A, P = inp.ISOTHERMAL, inp.ADIABATIC, inp.PERIODIC
SHAPES = [(2, 1, 1), (2, 3, 2), (16, 16, 3), (32, 4, 4), (80, 30, 4), (96, 5, 3), (130, 16, 2),
          (256, 1, 3), (33, 31, 3), (128, 2, 2)]


@pytest.mark.parametrize("shape", SHAPES)
@pytest.mark.parametrize("bc", [[I, A, A, I, I, A], [P, P, I, A, A, I], [A, I, P, P, P, P]])
@pytest.mark.parametrize("precision,streaming,tol", [
    (inp.FP32, inp.PULL, 5e-6), (inp.FP16, inp.PULL, 2.5e-4), (inp.FP32, inp.AA, 5e-6),
    (inp.FP64, inp.PULL, 1e-13)])
def test_one_step_at_the_edges_of_the_launch_shapes(shape, bc, precision, streaming, tol):
    p = inp.Params(precision=precision, streaming=streaming, Ra=5e4, Pr=0.5, St=0.7, bc=bc,
                   T_wall=[1.0, 0.1, 0.3, 0.8, 0.6, 0.2])
    f, gq = inp.random_state(shape, seed=11)
    dev = torch.device("cuda")
    g, o = LBPC(shape, p), oracle.Oracle(shape, p)
    g.set_distributions(torch.from_numpy(f).to(dev), torch.from_numpy(gq).to(dev))
    f0, g0 = g.distributions()
    o.set_distributions(f0.cpu().numpy(), g0.cpu().numpy())
    for _ in range(2):  # AA: an even and an odd step
        g.step(1)
        o.step(1)
        f1, g1 = (v.cpu().numpy() for v in g.distributions())
        fo, go = o.distributions()
        assert np.abs(f1 - fo).max() <= tol
        assert np.abs(g1[1:] - go[1:]).max() <= tol
        assert np.abs(g1[0] - go[0]).max() <= 6 * tol
        o.set_distributions(f1, g1)


@pytest.mark.parametrize("flow_model,precision,shapes", [
    # below, at and above the largest lattice that is stepped in blocks
    (inp.FLOW_MRT, inp.FP32, [(1, 1, 1), (7, 9, 65), (64, 8, 16), (64, 8, 17)]),
    (inp.FLOW_SRT, inp.FP32, [(24, 12, 10)]),
    (inp.FLOW_MRT, inp.FP64, [(3, 2, 5), (8, 8, 8), (9, 8, 8)]),
    (inp.FLOW_NONE, inp.FP64, [(64, 4, 4), (16, 16, 16)]),
    (inp.FLOW_NONE, inp.FP32, [(6, 1, 40), (128, 1, 64)]),
    (inp.FLOW_NONE, inp.FP16, [(94, 4, 9)]), (inp.FLOW_NONE, inp.BF16, [(39, 1, 11)]),
    (inp.FLOW_NONE, inp.FP16_G32, [(39, 1, 11)]), (inp.FLOW_MRT, inp.FP16, [(24, 12, 10)]),
    (inp.FLOW_MRT, inp.BF16_G32, [(25, 12, 10)])])
@pytest.mark.parametrize("streaming", [inp.PULL, inp.AA])
def test_blocks_of_steps_equal_single_steps(flow_model, precision, shapes, streaming):
    for shape in shapes:
        for bc in ([I, A, A, I, I, A], [I, I, P, P, A, A]):
            p = inp.Params(flow_model=flow_model, precision=precision, streaming=streaming, bc=bc,
                           Ra=1e5, Pr=0.7, tau_g=0.0 if flow_model else 0.9, report_every=9,
                           T_wall=[1.0, 0.1, 0.3, 0.8, 0.6, 0.2])
            h0 = np.random.default_rng(2).uniform(-0.3, 1.8, int(np.prod(shape)))
            a, b = LBPC(shape, p), LBPC(shape, p)
            for v in (a, b):
                v.set_initial_h(h0)
            a.step(23)
            a.step(8)  # from an odd step on
            for _ in range(31):
                b.step(1)
            for k, v in a.fields().items():
                assert torch.equal(v, b.fields()[k]), (shape, bc, k)
            assert np.array_equal(a.history(), b.history()), (shape, bc)
            if streaming == inp.PULL:
                assert a.save() == b.save(), (shape, bc)


@pytest.mark.parametrize("shape,precision,flow_model,streaming", [
    ((64, 16, 16), inp.FP32, inp.FLOW_MRT, inp.PULL), ((16, 8, 8), inp.FP32, inp.FLOW_MRT, inp.PULL),
    ((64, 4, 4), inp.FP64, inp.FLOW_NONE, inp.PULL), ((24, 24, 24), inp.FP64, inp.FLOW_MRT, inp.PULL),
    ((33, 16, 16), inp.FP16, inp.FLOW_MRT, inp.AA), ((16, 8, 8), inp.FP32, inp.FLOW_MRT, inp.AA)])
def test_captured_steps_can_be_replayed(shape, precision, flow_model, streaming):
    """An even number of steps recorded into a CUDA graph, replayed, equals the same calls."""
    p = inp.Params(precision=precision, flow_model=flow_model, streaming=streaming, Ra=1e5, Pr=0.7,
                   tau_g=0.0 if flow_model else 0.8, report_every=10 ** 6)
    h0 = np.random.default_rng(0).uniform(-0.2, 1.5, int(np.prod(shape)))
    s = torch.cuda.Stream()
    with torch.cuda.stream(s):
        a, b = LBPC(shape, p, stream=s), LBPC(shape, p, stream=s)
        for v in (a, b):
            v.set_initial_h(h0)
            v.step(6)
        s.synchronize()
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph, stream=s):
            a.step(6)
        for _ in range(3):
            graph.replay()
            b.step(6)
        A, R = a.fields(), b.fields()
        s.synchronize()
        for k, v in A.items():
            assert torch.equal(v, R[k]), k
