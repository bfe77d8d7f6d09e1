"""The server admits lattices by footprint_bytes: what a lattice with a table on every face
holds on the device once it has formed a residual."""
import pytest

import lbm_inputs as inp

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec", ["f64", "f32", "f16"])
@pytest.mark.parametrize("scheme", ["ab", "aa"])
@pytest.mark.parametrize("dims", [(5, 4, 3), (97, 64, 64)])  # one row of partial sums, and more than 1,024
def test_footprint_is_what_a_lattice_holds(prec, scheme, dims):
    import paper_0811_4593_gb300 as lbm
    from paper_0811_4593_gb300.serving import footprint_bytes
    wl = inp.random_face_workload(7, *dims, 0.9, (False, False, False))
    assert all(t is not None for t in wl.utabs)
    with lbm.Lattice.from_workload(wl, prec, scheme=scheme) as lat:
        lat.residual()
        assert lat.info()["device_bytes"] == footprint_bytes(*dims, prec, scheme)
