"""A geometry set when device memory is short: with no room for the list of fluid nodes the
lattice steps without it, and a geometry that is refused leaves the lattice as it was."""
import ctypes as C

import numpy as np
import pytest

import lbm_inputs as inp
from lbm_testlib import encode, noisy_state

pytestmark = pytest.mark.gpu


@pytest.fixture
def refuse():
    """The sizes (bytes per node) that the allocator turns down."""
    import torch

    from paper_0811_4593_gb300 import _binding as b
    sizes, held, prev = set(), {}, b._hooks

    def alloc(nbytes, _user):
        if nbytes - 512 in sizes:  # 256 guard bytes at either end
            return None
        t = torch.empty(int(nbytes), dtype=torch.uint8, device="cuda")
        held[t.data_ptr()] = t
        return t.data_ptr()

    def free(p, _user):
        del held[p]

    hooks = (C.CFUNCTYPE(C.c_void_p, C.c_size_t, C.c_void_p)(alloc),
             C.CFUNCTYPE(None, C.c_void_p, C.c_void_p)(free))
    b.check(b.lib().lbm_set_allocator(C.cast(hooks[0], C.c_void_p), C.cast(hooks[1], C.c_void_p), None))
    b._hooks = hooks
    yield sizes
    b._hooks = prev
    if prev:
        b.check(b.lib().lbm_set_allocator(C.cast(prev[0], C.c_void_p), C.cast(prev[1], C.c_void_p), None))
    else:
        b.use_default_allocator()


@pytest.mark.parametrize("prec", ["f64", "f32", "f16"])
def test_a_geometry_without_room_for_its_list(prec, refuse):
    import paper_0811_4593_gb300 as lbm
    wl = inp.channel(33, 19, 21, 0.9, (0.02, 0.01, 0.0))
    shape = (19, wl.nz, wl.ny, wl.nx)
    n = wl.nx * wl.ny * wl.nz
    s0 = encode(noisy_state(shape, 6, u=(0.01, -0.004, 0.006)), prec)
    solid = [(inp.noise(seed, shape[1:]) > 0.5).astype(np.uint8) for seed in (5, 6)]
    with lbm.Lattice.from_workload(wl, prec) as lat, lbm.Lattice.from_workload(wl, prec) as ref:
        for l in (lat, ref):
            l.set_populations(s0)
            l.step(3)
        refuse.add(4 * n)  # no words, no geometry: the lattice goes on without one
        with pytest.raises(lbm.LBMError):
            lat.set_solid(solid[0])
        refuse.clear()
        for l in (lat, ref):
            l.step(3)
        np.testing.assert_array_equal(lat.get_populations(), ref.get_populations())
        for mask in solid:
            refuse.add(8 * n)
            lat.set_solid(mask)
            refuse.clear()
            ref.set_solid(mask)
            for steps in (1, 17):
                for l in (lat, ref):
                    l.step(steps)
                np.testing.assert_array_equal(lat.get_populations(), ref.get_populations())
        lat.check_guards()
