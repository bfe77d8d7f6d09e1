"""The residual sums of float and binary16 lattices against exact rational arithmetic on the
stored velocities: no further off than sums formed in double throughout."""
import ctypes as C
from fractions import Fraction

import numpy as np
import pytest

import lbm_inputs as inp
from lbm_testlib import encode, noisy_state

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec", ["f32", "f16"])
@pytest.mark.parametrize("dims", [(3, 3, 3), (4, 4, 68), (17, 13, 12)])
def test_sums_of_squares_are_those_of_double(prec, dims):
    import torch

    import paper_0811_4593_gb300 as lbm
    nx, ny, nz = dims
    n = nx * ny * nz
    snap = torch.zeros((3, nz, ny, nx), device="cuda")
    sums = torch.zeros(4, dtype=torch.float64, device="cuda")
    # roundings in double behind the exact warp sums, each at most 2^-53 of its result: one to
    # double, and where there are more warps and blocks the adds of the block and of the fold
    blocks = (n + 255) // 256
    roundings = 1 if n <= 32 else 1 + 3 + (0 if blocks == 1 else 3 + 5 + 3)
    for seed in range(12):
        state = encode(noisy_state((19, nz, ny, nx), seed, amp=0.05, u=(0.03, -0.02, 0.01)), prec)
        before = 0.05 * inp.noise(100 + seed, tuple(snap.shape)).astype(np.float32)
        snap.copy_(torch.from_numpy(before))
        pops = torch.from_numpy(state).cuda()
        st = lbm.lib().lbm_reduce_state_static(C.c_void_p(pops.data_ptr()), nx, ny, nz, 1 if prec == "f32" else 2, 1.0,
                                               C.c_void_p(snap.data_ptr()), C.c_void_p(sums.data_ptr()),
                                               C.c_void_p(torch.cuda.current_stream().cuda_stream))
        assert st == 0
        got = sums.cpu().numpy()
        u = [Fraction(float(v)) for v in snap.cpu().numpy().ravel()]
        p = [Fraction(float(v)) for v in before.ravel()]
        for k, exact in ((1, sum((a - b) ** 2 for a, b in zip(u, p))), (2, sum(a * a for a in u))):
            off = abs(float((Fraction(float(got[k])) - exact) / exact))
            assert off <= (roundings + 0.01) * 2.0 ** -53, (seed, k, off * 2.0 ** 53)
