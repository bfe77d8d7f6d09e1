"""Long runs of lattices with solid nodes, too large for the multi-step kernels: one launch for
each step, the bits of steps taken one call each, and solid populations kept."""
import numpy as np
import pytest

import lbm_inputs as inp
from lbm_testlib import encode, noisy_state

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec", ["f64", "f32", "f16"])
@pytest.mark.parametrize("above", [0.5, 0.95])  # a quarter and a fortieth: with and without a list
def test_long_runs_by_launches(prec, above):
    import torch

    import paper_0811_4593_gb300 as lbm
    nodes = torch.cuda.get_device_properties(0).multi_processor_count * (512 if prec == "f64" else 1024)
    wl = inp.channel(61, 47, 2 * nodes // (61 * 47), 0.9, (0.02, 0.01, 0.0))
    shape = (19, wl.nz, wl.ny, wl.nx)
    solid = inp.noise(5, shape[1:]) > above
    wl.solid = solid.astype(np.uint8)
    s0 = encode(noisy_state(shape, 6, u=(0.01, -0.004, 0.006)), prec)
    with lbm.Lattice.from_workload(wl, prec) as lat, lbm.Lattice.from_workload(wl, prec) as one:
        for l in (lat, one):
            l.set_populations(s0)
        for n in (17, 20):
            before = lat.info()["kernel_launches"]
            lat.step(n)
            assert lat.info()["kernel_launches"] - before == n
            for _ in range(n):
                one.step(1)
            got = lat.get_populations()
            np.testing.assert_array_equal(got, one.get_populations())
            np.testing.assert_array_equal(got[:, solid], s0[:, solid])
        lat.check_guards()
