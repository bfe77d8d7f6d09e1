"""Plain steps do not touch solid nodes: their populations survive steps of every kind and
loads of part of the state, in whichever array holds it."""
import numpy as np
import pytest

import lbm_inputs as inp
from lbm_testlib import encode, noisy_state

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec", ["f64", "f32", "f16"])
@pytest.mark.parametrize("above", [0.5, 0.9, -1.1])
@pytest.mark.parametrize("dims", [(17, 13, 12), (33, 19, 21)])
def test_solid_populations_are_kept(prec, dims, above):
    # a quarter, a twentieth and all of the nodes solid (with and without a list of the fluid
    # ones); 2,652 nodes (one launch for a long run) and 13,167 (one launch per step); a slab of
    # the state is replaced between odd and even numbers of steps
    import paper_0811_4593_gb300 as lbm
    wl = inp.channel(*dims, 0.9, (0.02, 0.01, 0.0))
    shape = (19, wl.nz, wl.ny, wl.nx)
    solid = inp.noise(5, shape[1:]) > above
    wl.solid = solid.astype(np.uint8)
    s = [encode(noisy_state(shape, seed, u=(0.01, -0.004, 0.006)), prec) for seed in (6, 7, 8)]
    with lbm.Lattice.from_workload(wl, prec) as lat:
        lat.set_populations(s[0])
        held = s[0].copy()
        for i, n in enumerate((1, 16, 3, 17, 2, 20)):
            lat.step(n)
            np.testing.assert_array_equal(lat.get_populations()[:, solid], held[:, solid])
            part = s[1 + i % 2][:, 2:7]
            lat.set_populations(part, z0=2)
            held[:, 2:7] = part
            lat.step_residual(1 + i % 2)
            np.testing.assert_array_equal(lat.get_populations()[:, solid], held[:, solid])
        lat.check_guards()
