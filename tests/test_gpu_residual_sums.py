"""The residual sums at the edges of their ranges: velocities below and above what the
float-pair sums cover, a block with a single node, and lattices on both sides of one fold
group (1024 blocks of 256 nodes)."""
import numpy as np
import pytest

import lbm_inputs as inp
from lbm_testlib import decode, encode, noisy_state

pytestmark = pytest.mark.gpu


def _velocities(wl, stored, prec):
    """Density deviation and velocity of stored populations, in double."""
    import oracle
    c, w, _ = oracle.lattice()
    f = stored.astype(np.float64)
    drho = f.sum(0) - (1.0 if prec == "f64" else 0.0)
    j = np.tensordot(np.asarray(c, np.float64).T, f, 1)
    return drho, j / (1.0 + drho)


@pytest.mark.parametrize("prec", ["f64", "f32"])
@pytest.mark.parametrize("scales", [(1e-30, 1e-30), (1e-30, 1e-3), (1e-3, 1e12), (0.0, 1e-3), (1e-24, 0.0)])
def test_velocities_of_any_size(prec, scales):
    # half of the nodes have velocities of one size, half of the other; FP64 stores f, in
    # which velocities below 1e-16 are lost, so it takes the larger ones only
    import paper_0811_4593_gb300 as lbm
    if prec == "f64" and min(scales) < 1e-3:
        pytest.skip("not representable in f")
    wl = inp.make_workload("box", 13, 9, 11, 0.9, [None] * 6)
    shape = (19, 11, 9, 13)
    size = np.where(np.arange(11 * 9 * 13).reshape(shape[1:]) < 640, *scales)
    states = []
    for seed in (1, 2):
        h = inp.noise(seed, shape)
        h[18] = -h[:18].sum(0)  # no density deviation beyond rounding
        s = h * size
        states.append(s.astype(np.float32) if prec == "f32" else s + np.asarray(_weights())[:, None, None, None])
    with lbm.Lattice.from_workload(wl, prec) as lat:
        for k, s in enumerate(states):
            lat.set_populations(s)
            if k:
                # large velocities come with density deviations below zero: the sums are
                # compared through the call that returns them in either case
                try:
                    r, m = lat.residual()
                except lbm.LBMDiverged as e:
                    r, m = e.residual, e.mass
            else:
                try:
                    lat.residual()
                except lbm.LBMDiverged:
                    pass
    u = []
    for s in states:
        with lbm.Lattice.from_workload(wl, prec) as lat:
            lat.set_populations(s)
            rho, v = lat.macros()
            u.append(v.double().cpu().numpy())
            last = rho.double().cpu().numpy()
    want = np.sqrt(((u[1] - u[0]) ** 2).sum()) / np.sqrt((u[1] ** 2).sum())
    # the library's own float velocities, so only the sums are compared: pairs hold 2^-47
    assert r == pytest.approx(want, rel=1e-12)
    # the mass of float lattices sums the deviations, the densities here are rounded to float
    assert m == pytest.approx(last.sum(), rel=1e-13 if prec == "f64" else 1e-6, abs=1e-6 * np.abs(last).sum())


def _weights():
    import oracle
    return oracle.lattice()[1]


@pytest.mark.parametrize("prec", ["f64", "f32", "f16"])
@pytest.mark.parametrize("dims", [(3, 3, 3), (257, 3, 3), (128, 64, 32), (131, 64, 32)])
def test_fold_sizes_alone_and_in_a_batch(prec, dims):
    # 27 nodes (one ragged block), 2,313 (ten blocks), 262,144 (exactly one group of 1024
    # blocks) and 268,288 (two groups): the oracle's sums, and the same bits in a batch
    import oracle
    import paper_0811_4593_gb300 as lbm
    wl = inp.make_workload("box", *dims, 0.8, [None] * 6)
    shape = (19, dims[2], dims[1], dims[0])
    s = [encode(noisy_state(shape, seed, u=(0.02, 0.01, -0.01)), prec) for seed in (3, 4)]
    with lbm.Lattice.from_workload(wl, prec) as lat:
        lat.set_populations(s[0])
        lat.residual()
        lat.set_populations(s[1])
        r, m = lat.residual()
        lat.set_populations(s[0])
        alone = lat.step_residual(2)
    olat = oracle.Lattice.from_workload(wl)
    _, u0 = oracle.macros(olat, decode(s[0], prec))
    red = oracle.reduce(olat, decode(s[1], prec), u0)
    assert m == pytest.approx(red[0], rel=1e-12 if prec == "f64" else 1e-5)
    assert abs(r - np.sqrt(red[1]) / np.sqrt(red[2])) <= (1e-12 if prec == "f64" else 1e-5)
    with lbm.Lattice.from_workload(wl, prec) as lat, lbm.Batch(2, prec) as batch:
        lat.set_populations(s[1])
        lat.residual()
        lat.set_populations(s[0])
        batch.attach(1, lat)
        batch.step(2, residual=True)
        assert batch.results()[1] == (*alone, 0)
        batch.detach(1)
