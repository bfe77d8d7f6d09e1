"""Which lattices take pairs of steps in place: the ones whose single array fills 3/7 to 4/5 of
the L2 cache. Seen from the second population array, which pairs in place leave alone."""
import ctypes as C

import numpy as np
import pytest

import lbm_inputs as inp

pytestmark = pytest.mark.gpu


@pytest.fixture
def buffers():
    """The device buffers the library asks for, as byte tensors in the order of the requests."""
    import torch

    from paper_0811_4593_gb300 import _binding as b
    held, prev = {}, b._hooks

    def alloc(nbytes, _user):
        t = torch.empty(int(nbytes), dtype=torch.uint8, device="cuda")
        held[t.data_ptr()] = t
        return t.data_ptr()

    def free(p, _user):
        del held[p]

    hooks = (C.CFUNCTYPE(C.c_void_p, C.c_size_t, C.c_void_p)(alloc), C.CFUNCTYPE(None, C.c_void_p, C.c_void_p)(free))
    b.check(b.lib().lbm_set_allocator(C.cast(hooks[0], C.c_void_p), C.cast(hooks[1], C.c_void_p), None))
    b._hooks = hooks
    yield held
    b._hooks = prev
    if prev:
        b.check(b.lib().lbm_set_allocator(C.cast(prev[0], C.c_void_p), C.cast(prev[1], C.c_void_p), None))
    else:
        b.use_default_allocator()


def _in_place(wl, prec, buffers):
    import torch

    import paper_0811_4593_gb300 as lbm
    nbytes = 19 * wl.nx * wl.ny * wl.nz * {"f64": 8, "f32": 4, "f16": 2}[prec]
    with lbm.Lattice.from_workload(wl, prec) as lat:
        arrays = [t for t in buffers.values() if t.numel() == nbytes + 512]  # 256 guard bytes each side
        assert len(arrays) == 2
        lat.step(2)  # an even number: the state is in the first array again
        lat.sync()
        other = arrays[1][256:-256]
        other.fill_(0x5a)
        torch.cuda.synchronize()
        lat.step(4)
        lat.sync()
        return bool((other == 0x5a).all())


def _nz(fraction, row=64 * 64):
    import torch
    return fraction * torch.cuda.get_device_properties(0).L2_cache_size / (19 * 4 * row)


def test_the_range_of_pairs_in_place(buffers):
    low, high = int(np.ceil(_nz(3 / 7))), int(_nz(4 / 5))
    for nz, expected in ((low - 1, False), (low, True), ((low + high) // 2, True), (high, True), (high + 1, False)):
        assert _in_place(inp.make_workload("periodic", 64, 64, nz, 0.8, [None] * 6), "f32", buffers) == expected, nz


def test_other_lattices_use_both_arrays(buffers):
    nz = int(_nz(0.6))
    wl = inp.make_workload("periodic", 64, 64, nz, 0.8, [None] * 6)
    assert not _in_place(inp.make_workload("periodic", 64, 64, 2 * nz, 0.8, [None] * 6), "f16", buffers)
    assert not _in_place(inp.make_workload("periodic", 64, 64, nz // 2, 0.8, [None] * 6), "f64", buffers)
    wl.force = (0.0, 0.0, 1e-5)
    assert not _in_place(wl, "f32", buffers)
