"""The multi-step kernel with a grid barrier beside other work on the GPU: its blocks need not
find room at once, and the steps hold the bits of the same steps taken one call each."""
import threading

import numpy as np
import pytest

import lbm_inputs as inp
from lbm_testlib import encode, noisy_state

pytestmark = pytest.mark.gpu


def _whole_chip():
    """A lattice of 1,024 nodes for each SM (a block of it fills an SM's registers)."""
    import torch
    return inp.channel(32, 32, torch.cuda.get_device_properties(0).multi_processor_count, 0.8, (0.02, 0.01, 0.0))


def _solid(wl):
    wl.solid = (inp.noise(5, (wl.nz, wl.ny, wl.nx)) > 0.8).astype(np.uint8)
    return wl


@pytest.mark.parametrize("solid", [False, True])
def test_steps_beside_a_kernel_that_holds_an_sm(solid):
    # a foreign kernel takes an SM for about three times as long as any wait of the steps lasts
    import torch

    import paper_0811_4593_gb300 as lbm
    wl = _solid(_whole_chip()) if solid else _whole_chip()
    s0 = encode(noisy_state((19, wl.nz, wl.ny, wl.nx), 6), "f32")
    side = torch.cuda.Stream()
    with lbm.Lattice.from_workload(wl, "f32", stream=torch.cuda.Stream()) as lat, \
            lbm.Lattice.from_workload(wl, "f32") as ref:
        lat.step(16)  # the first launch of a kernel loads it, which waits for running ones
        lat.set_populations(s0)
        ref.set_populations(s0)
        for _ in range(20 + 33):
            ref.step(1)
        ref.sync()
        with torch.cuda.stream(side):
            torch.cuda._sleep(6_000_000_000)
        before = lat.info()["kernel_launches"]
        lat.step(20)
        lat.step(33)
        assert lat.info()["kernel_launches"] - before == 2
        assert not side.query()
        lat.sync()
        np.testing.assert_array_equal(lat.get_populations(), ref.get_populations())
        lat.check_guards()


@pytest.mark.parametrize("wl,scheme", [(inp.duct(29, 17, 16, 0.8, 0.05, 30.0), "ab"),
                                       (inp.duct(29, 17, 16, 0.8, 0.05, 30.0), "aa"),
                                       (inp.duct(45, 23, 21, 0.8, 0.05, 30.0), "ab")], ids=["cluster", "cluster_aa", "grid"])
def test_long_runs_give_way_to_other_work(wl, scheme):
    # no launch holds its SMs for more than 4,096 steps; the rest follows in the same ways
    import paper_0811_4593_gb300 as lbm
    with lbm.Lattice.from_workload(wl, "f32", scheme=scheme) as lat, lbm.Lattice.from_workload(wl, "f32") as ref:
        for n, launches in ((4096, 1), (4112, 2), (8192 + 6, 2 + 6)):
            before = lat.info()["kernel_launches"]
            lat.step(n)
            assert lat.info()["kernel_launches"] - before == launches
            for _ in range(n // 2):
                ref.step(2)
            np.testing.assert_array_equal(lat.get_populations(), ref.get_populations())


def test_two_threads_step_lattices_that_cover_the_chip():
    import torch

    import paper_0811_4593_gb300 as lbm
    wl = _whole_chip()
    steps, calls, failed, got = 400, 50, [], []
    s0 = encode(noisy_state((19, wl.nz, wl.ny, wl.nx), 6), "f32")

    def advance(gate):
        try:
            with lbm.Lattice.from_workload(wl, "f32", stream=torch.cuda.Stream()) as lat:
                lat.set_populations(s0)
                gate.wait()
                for _ in range(calls):
                    lat.step(steps)
                lat.sync()
                got.append(lat.get_populations())
        except BaseException as e:  # noqa: BLE001 - handed to the main thread
            failed.append(e)

    for parties in (1, 2):
        gate = threading.Barrier(parties, timeout=60)
        threads = [threading.Thread(target=advance, args=(gate,)) for _ in range(parties)]
        for t in threads:
            t.start()
        for t in threads:
            t.join()
    assert not failed, failed
    np.testing.assert_array_equal(got[1], got[0])
    np.testing.assert_array_equal(got[2], got[0])
