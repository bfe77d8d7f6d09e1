"""A/B lattices whose single array fits in L2 take pairs of steps in place: the bits of single
steps, which alternate the two arrays, for even and odd counts, beside the residual and on
both sides of the range."""
import pytest

import lbm_inputs as inp

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("wl", [inp.duct(256, 56, 56, 0.7, 0.05, 30.0),             # 61 MB
                                inp.channel(101, 83, 110, 0.8, (0.03, 0.01, 0.0)),  # 70 MB, odd rows
                                inp.pressure_duct(100, 100, 1.0),                   # 76 MB, pressure planes
                                inp.make_workload("periodic", 96, 96, 128, 0.6, [None] * 6),    # 90 MB
                                inp.channel(128, 64, 64, 0.8, (0.03, 0.01, 0.0)),   # 40 MB: two arrays
                                inp.channel(256, 96, 64, 0.8, (0.03, 0.01, 0.0))],  # 120 MB: two arrays
                         ids=lambda w: f"{w.name}_{w.nx}x{w.ny}x{w.nz}")
def test_pairs_in_place_equal_single_steps(wl):
    import torch

    import paper_0811_4593_gb300 as lbm
    gen = torch.Generator("cuda").manual_seed(3)
    s0 = 1e-3 * (torch.rand((19, wl.nz, wl.ny, wl.nx), generator=gen, device="cuda") - 0.5)
    a_pops, b_pops = torch.empty_like(s0), torch.empty_like(s0)
    with lbm.Lattice.from_workload(wl, "f32") as a, lbm.Lattice.from_workload(wl, "f32") as b:
        for lat in (a, b):
            lat.set_populations(s0)
        for n in (2, 5, 1, 4):
            a.step(n)
            for _ in range(n):
                b.step(1)
            assert torch.equal(a.get_populations(out=a_pops), b.get_populations(out=b_pops))
        for n in (6, 7):
            ra = a.step_residual(n)
            for _ in range(n - 1):
                b.step(1)
            assert ra == b.step_residual(1)
            assert torch.equal(a.get_populations(out=a_pops), b.get_populations(out=b_pops))
        a.check_guards()
