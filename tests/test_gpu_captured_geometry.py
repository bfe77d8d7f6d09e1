"""Steps captured in a CUDA graph replay with the geometry last set, whatever number of fluid
nodes the lattice had when they were captured."""
import numpy as np
import pytest

import lbm_inputs as inp
from lbm_testlib import encode, noisy_state

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dims,n", [((17, 13, 12), 16), ((33, 19, 21), 16), ((33, 19, 21), 2)],
                         ids=["cluster", "grid", "launches"])
def test_replays_follow_the_geometry(dims, n):
    import torch

    import paper_0811_4593_gb300 as lbm
    wl = inp.channel(*dims, 0.9, (0.02, 0.01, 0.0))
    shape = (19, wl.nz, wl.ny, wl.nx)
    s0 = encode(noisy_state(shape, 6, u=(0.01, -0.004, 0.006)), "f32")
    noise = inp.noise(5, shape[1:])
    stream = torch.cuda.Stream()
    with lbm.Lattice.from_workload(wl, "f32", stream=stream) as lat, lbm.Lattice.from_workload(wl, "f32") as ref:
        for l in (lat, ref):
            l.set_populations(s0)
            l.set_solid((noise > 0.0).astype(np.uint8))  # half of the nodes
            l.step(n)
        lat.sync()
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph, stream=stream):
            lat.step(n)
        for above in (0.0, 0.7, -0.6, 0.95, 0.3):  # more, fewer, too few solid nodes for a list
            solid = (noise > above).astype(np.uint8)
            for l in (lat, ref):
                l.set_solid(solid)
            graph.replay()
            torch.cuda.synchronize()
            for _ in range(n):
                ref.step(1)
            np.testing.assert_array_equal(lat.get_populations(), ref.get_populations())
        lat.check_guards()
