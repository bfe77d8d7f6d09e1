"""Two host threads that step a lattice each at the same time: every call succeeds, takes the
route it takes alone, and the states hold the bits of the same runs alone."""
import threading

import numpy as np
import pytest

import lbm_inputs as inp
from lbm_testlib import encode, noisy_state

pytestmark = pytest.mark.gpu


def _periodic(nx, ny, nz):
    return inp.make_workload("periodic", nx, ny, nz, 0.7, [None] * 6)


# lattices of one kernel whose launches need unlike amounts of shared memory
PAIRS = {
    "cluster_f64": ("f64", _periodic(16, 16, 16), _periodic(3, 3, 3), 16),
    "cluster_f32": ("f32", _periodic(32, 16, 16), _periodic(3, 3, 3), 16),
    "cluster_f16": ("f16", _periodic(32, 16, 16), _periodic(3, 3, 3), 16),
    "rows_f16": ("f16", _periodic(2048, 3, 3), _periodic(264, 3, 3), 2),
}


@pytest.mark.parametrize("name", list(PAIRS))
def test_two_threads_step_lattices_of_unlike_sizes(name):
    import torch

    import paper_0811_4593_gb300 as lbm
    prec, *wls, n = PAIRS[name]
    calls, failed = 1500, []

    def advance(wl, out, gate=None):
        try:
            with lbm.Lattice.from_workload(wl, prec, stream=torch.cuda.Stream()) as lat:
                lat.set_populations(encode(noisy_state((19, wl.nz, wl.ny, wl.nx), 6, amp=0.005), prec))
                before = lat.info()["kernel_launches"]
                if gate:
                    gate.wait()
                for _ in range(calls):
                    lat.step(n)
                out.append((lat.info()["kernel_launches"] - before, lat.get_populations()))
        except BaseException as e:  # noqa: BLE001 - handed to the main thread
            failed.append(e)

    alone = []
    for wl in wls:
        advance(wl, alone)
    gate = threading.Barrier(2, timeout=60)
    both = [[], []]
    threads = [threading.Thread(target=advance, args=(wl, out, gate)) for wl, out in zip(wls, both)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not failed, failed
    for (launches, state), ((launches_both, state_both),) in zip(alone, both):
        assert launches_both == launches
        np.testing.assert_array_equal(state_both, state)
