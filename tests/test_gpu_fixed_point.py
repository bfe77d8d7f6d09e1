"""FP64 nodes inside and outside the windows of the fixed-point relaxation, mixed in one
lattice: one step against the oracle, node by node, for density scales on both sides of a
power of two and with the sweep's variants giving the same bits."""
import numpy as np
import pytest

import lbm_inputs as inp

pytestmark = pytest.mark.gpu


def _state(seed, shape, rho0, mix):
    import oracle
    w = oracle.lattice()[1]
    f = (w * rho0)[:, None, None, None] * (1.0 + 0.2 * inp.noise(seed, shape))
    if mix:
        # whole nodes scaled by 2^-14 .. 2^6, single populations by 2^-8 .. 2^2, some of
        # either sign
        nodes = shape[1:]
        f *= np.exp2(-4.0 + 10.0 * inp.noise(seed + 1, nodes)) ** (inp.noise(seed + 2, nodes) > 0.4)
        f *= np.exp2(-3.0 + 5.0 * inp.noise(seed + 3, shape)) ** (inp.noise(seed + 4, shape) > 0.9)
        f[3] *= np.where(inp.noise(seed + 5, nodes) > 0.95, -1.0, 1.0)
    return f


@pytest.mark.parametrize("rho0,tau", [(1.0, 0.6), (1.0, 1.0), (0.999, 2.0), (3e8, 0.8), (1e-290, 0.8)])
@pytest.mark.parametrize("mix", [False, True])
def test_one_step_matches_the_oracle(rho0, tau, mix):
    import oracle
    import paper_0811_4593_gb300 as lbm
    wl = inp.make_workload("box", 33, 11, 9, tau, [None] * 6, rho0=rho0)
    shape = (19, 9, 11, 33)
    f0 = _state(11, shape, rho0, mix)
    out = {}
    for name in ("plain", "residual", "aa", "batch"):
        scheme = "aa" if name == "aa" else "ab"
        with lbm.Lattice.from_workload(wl, "f64", scheme=scheme) as lat:
            lat.set_populations(f0)
            if name == "residual":
                for _ in range(2):
                    try:
                        lat.step_residual(1)
                    except lbm.LBMDiverged:
                        pass
            elif name == "batch":
                with lbm.Batch(1, "f64") as batch:
                    batch.attach(0, lat)
                    batch.step(2)
                    batch.detach(0)
            else:
                lat.step(2)
            out[name] = lat.get_populations()
    for name in ("residual", "aa", "batch"):
        np.testing.assert_array_equal(out[name], out["plain"], err_msg=name)
    olat = oracle.Lattice.from_workload(wl)
    with lbm.Lattice.from_workload(wl, "f64") as lat:
        lat.set_populations(f0)
        lat.step(1)
        got = lat.get_populations()
    ref = oracle.run(olat, f0, 1)
    streamed = np.empty_like(f0)
    c = np.asarray(oracle.lattice()[0], int)
    for k in range(19):
        streamed[k] = np.roll(f0[k], tuple(c[k][::-1]), (0, 1, 2))
    # about 60 roundings of numbers no larger than the sum of the node's magnitudes, times
    # its momentum over its density where populations of both signs cancel in the latter
    size = np.abs(streamed).sum(0)
    grow = np.maximum(1.0, size / np.maximum(np.abs(streamed.sum(0)), 1e-300)) ** 2
    assert np.all(np.abs(got - ref) <= 60 * 2.0 ** -53 * size * grow)


def _solid():
    wl = inp.channel(19, 16, 17, 0.9, (0.03, 0.01, 0.0))
    wl.solid = (inp.noise(5, (17, 16, 19)) > 0.6).astype(np.uint8)
    return wl


CLOSURES = {
    "faces": lambda: inp.random_face_workload(51, 13, 10, 9, 0.8, (False, False, False)),
    "faces_beyond_a_quarter": lambda: inp.random_face_workload(52, 13, 10, 9, 1.0, (False, False, False), amp=0.4),
    "x_rows_of_three": lambda: inp.random_face_workload(53, 3, 17, 11, 0.9, (False, True, False)),
    "pressure": lambda: inp.random_pressure_workload(54, 12, 9, 11, 0.9),
    "pressure_far_off": lambda: inp.random_pressure_workload(55, 12, 9, 11, 0.9, periodic_y=True, amp=0.9),
    "embedded": lambda: inp.embedded_walls(inp.make_workload("box", 9, 8, 7, 0.8, [inp.ZERO] * 6)),
    "pillar_x": lambda: inp.pillar_channel(axis=0, flow=1),
    "pillar_y": lambda: inp.pillar_channel(axis=1, flow=0),
    "pillar_z": lambda: inp.pillar_channel(axis=2, flow=1, force=3e-3),
    "solid": _solid,
}


@pytest.mark.parametrize("mix", [False, True])
@pytest.mark.parametrize("name", list(CLOSURES))
def test_closures_match_the_oracle(name, mix):
    # every face, edge, corner and geometry rule, with prescribed values on both sides of
    # what the fixed-point closures take, on states inside and partly outside the windows
    import oracle
    import paper_0811_4593_gb300 as lbm
    wl = CLOSURES[name]()
    shape = (19, wl.nz, wl.ny, wl.nx)
    w = oracle.lattice()[1][:, None, None, None]
    f0 = w * (1.0 + 0.1 * inp.noise(21, shape))
    if mix:
        f0 *= np.exp2(-2.0 + 3.0 * inp.noise(22, shape)) ** (inp.noise(23, shape) > 0.9)
    with lbm.Lattice.from_workload(wl, "f64") as lat:
        lat.set_populations(f0)
        lat.step(1)
        got = lat.get_populations()
        lat.check_guards()
    ref = oracle.run(oracle.Lattice.from_workload(wl), f0, 1)
    # about 100 roundings of numbers no larger than the neighbourhood's populations, times
    # 1 / (1 - u.n) <= 5/3 of a closure and its square in the equilibrium; a pressure plane
    # of density 0.1 next to density 1 has |u| near 1, squared over 0.1
    size = max(np.abs(f0).sum(0).max(), np.abs(ref).sum(0).max())
    assert np.abs(got - ref).max() <= 100 * 2.0 ** -53 * size * (10.0 if "far" in name else 3.0)
