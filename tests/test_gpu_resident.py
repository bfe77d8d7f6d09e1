"""The multi-step kernels of small lattices: many steps in one call hold the bits of the same
steps taken one call each, for every rule, precision and scheme, at the edges of their node
ranges (32 nodes per CTA or fewer, ragged last CTAs, 4,096 and 8,192 nodes, 512 and 1,024
nodes per SM of 152, and one node row more), and a grid barrier that runs out is reported."""
import numpy as np
import pytest

import lbm_inputs as inp
from lbm_testlib import encode, noisy_state

pytestmark = pytest.mark.gpu

WORKLOADS = {
    "27_nodes": lambda: inp.random_face_workload(41, 3, 3, 3, 1.0, (False, False, False)),
    "couette": lambda: inp.couette(),
    "pressure": lambda: inp.random_pressure_workload(42, 13, 9, 7, 0.9),
    "duct": lambda: inp.duct(29, 17, 16, 0.8, 0.05, 30.0),
    "8192_nodes": lambda: inp.make_workload("periodic", 32, 16, 16, 0.7, [None] * 6),
    "8208_nodes": lambda: inp.make_workload("periodic", 27, 19, 16, 0.7, [None] * 6),
    "4096_nodes": lambda: inp.channel(16, 16, 16, 0.7, (0.02, 0.01, 0.0)),
    "4112_nodes": lambda: inp.channel(257, 4, 4, 0.7, (0.02, 0.01, 0.0)),
    "grid_duct": lambda: inp.duct(45, 23, 21, 0.8, 0.05, 30.0),
    "grid_pressure": lambda: inp.random_pressure_workload(43, 33, 19, 17, 0.9),
    "grid_pillar": lambda: inp.pillar_channel(n=(41, 33, 12)),
    "77824_nodes": lambda: inp.couette(64, 32, 38),
    "79872_nodes": lambda: inp.couette(64, 32, 39),
    "155648_nodes": lambda: inp.couette(64, 32, 76),
    "157696_nodes": lambda: inp.couette(64, 32, 77),
    "pillar": lambda: inp.pillar_channel(),
    "force": lambda: inp.force_poiseuille(16, 1.2, 1e-5),
}


def _solid(wl):
    wl.solid = (inp.noise(5, (wl.nz, wl.ny, wl.nx)) > 0.7).astype(np.uint8)
    return wl


WORKLOADS["solid"] = lambda: _solid(inp.channel(17, 13, 12, 0.9, (0.02, 0.01, 0.0)))


@pytest.mark.parametrize("prec", ["f64", "f32", "f16"])
@pytest.mark.parametrize("name", list(WORKLOADS))
def test_one_call_equals_single_steps(name, prec):
    import paper_0811_4593_gb300 as lbm
    wl = WORKLOADS[name]()
    s0 = encode(noisy_state((19, wl.nz, wl.ny, wl.nx), 6, u=(0.01, -0.004, 0.006)), prec)
    schemes = ["ab"] if wl.solid is not None or wl.force is not None else ["ab", "aa"]
    for scheme in schemes:
        with lbm.Lattice.from_workload(wl, prec, scheme=scheme) as many, lbm.Lattice.from_workload(wl, prec) as one:
            many.set_populations(s0)
            one.set_populations(s0)
            for n in ((17, 16, 33) if scheme == "ab" else (16, 18)):
                l0 = many.info()["kernel_launches"]
                many.step(n)
                limit = (4096 if prec == "f64" else 8192) if scheme == "aa" else 152 * (512 if prec == "f64" else 1024)
                assert (many.info()["kernel_launches"] - l0 == 1) == (many.cells <= limit)
                for _ in range(n):
                    one.step(1)
                np.testing.assert_array_equal(many.get_populations(), one.get_populations())
            n = 20 if scheme == "ab" else 18
            for _ in range(n - 1):
                one.step(1)
            assert many.step_residual(n) == one.step_residual(1)
            np.testing.assert_array_equal(many.get_populations(), one.get_populations())
            many.check_guards()


def test_a_grid_barrier_that_runs_out_is_reported_and_the_context_recovers():
    import paper_0811_4593_gb300 as lbm
    wl = inp.channel(33, 20, 21, 0.8, (0.02, 0.01, 0.0))
    s0 = encode(noisy_state((19, wl.nz, wl.ny, wl.nx), 6), "f32")
    with lbm.Lattice.from_workload(wl, "f32") as lat, lbm.Lattice.from_workload(wl, "f32") as ref:
        assert lbm.lib().lbm_debug_drop_staged_copies(lat.ctx, 1) == 0
        lat.set_populations(s0)
        lat.step(16)
        with pytest.raises(lbm.LBMError, match="gave up waiting"):
            lat.sync()
        assert lbm.lib().lbm_debug_drop_staged_copies(lat.ctx, 0) == 0
        lat.sync()
        for l in (lat, ref):
            l.set_populations(s0)
            l.step(20)
        np.testing.assert_array_equal(lat.get_populations(), ref.get_populations())


@pytest.mark.parametrize("wl,prec,n", [(inp.couette(), "f64", 20), (inp.couette(), "f32", 2),
                                       (inp.channel(33, 20, 21, 0.8, (0.02, 0.01, 0.0)), "f32", 18),
                                       (inp.channel(256, 56, 56, 0.8, (0.02, 0.01, 0.0)), "f32", 4),
                                       (inp.channel(256, 9, 7, 0.8, (0.02, 0.01, 0.0)), "f16", 4)],
                         ids=["cluster", "launches", "grid", "in_place", "rows"])
def test_captured_steps_replay(wl, prec, n):
    # an even number of steps captured once and replayed: the state of as many steps
    import torch

    import paper_0811_4593_gb300 as lbm
    s0 = encode(noisy_state((19, wl.nz, wl.ny, wl.nx), 6, amp=0.005), prec)
    stream = torch.cuda.Stream()
    with lbm.Lattice.from_workload(wl, prec, stream=stream) as lat, lbm.Lattice.from_workload(wl, prec) as ref:
        for l in (lat, ref):
            l.set_populations(s0)
            l.step(n)
        lat.sync()
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph, stream=stream):
            lat.step(n)
        for _ in range(3):
            graph.replay()
        torch.cuda.synchronize()
        for _ in range(3):
            ref.step(n)
        np.testing.assert_array_equal(lat.get_populations(), ref.get_populations())
