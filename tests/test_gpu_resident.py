"""The multi-step kernel of small lattices: many steps in one call hold the bits of the same
steps taken one call each, for every rule, precision and scheme, at the edges of its node
range (32 nodes per CTA or fewer, ragged last CTAs, 8,192 nodes, and one node row more)."""
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
                assert (many.info()["kernel_launches"] - l0 == 1) == (many.cells <= 8192)
                for _ in range(n):
                    one.step(1)
                np.testing.assert_array_equal(many.get_populations(), one.get_populations())
            n = 20 if scheme == "ab" else 18
            for _ in range(n - 1):
                one.step(1)
            assert many.step_residual(n) == one.step_residual(1)
            np.testing.assert_array_equal(many.get_populations(), one.get_populations())
            many.check_guards()
