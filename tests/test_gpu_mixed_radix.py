"""Mixed-radix FFT passes: every radix of the schedules, two and three stages,
along each axis, in FP32, FP64 and float-float, against the FP64 oracle."""
import math

import numpy as np
import pytest

from oracle import bloch_oracle as O
from paper_2106_12487_gb300 import synth

pytestmark = pytest.mark.gpu
# FP32: a handful of roundings (2^-24 each) per stage of at most 3 stages and two
# directions on white noise stays below 5e-6 (the operator tolerance of the op
# tests); FP64 and float-float (48 bits) below 1e-12 likewise
TOL = {0: 1e-12, 1: 5e-6, 2: 1e-12}

# end radices 1..10, 12, 14, 15, 16 and middle radices 2..8 all occur
LENGTHS = [1, 2, 7, 14, 15, 27, 49, 90, 98, 120, 125, 140, 168, 210, 240, 243, 256, 343, 486, 512]


@pytest.fixture(scope="module")
def B():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2106_12487_gb300 import bloch, build
    build.build()
    bloch.lib()
    return bloch


@pytest.mark.parametrize("axis", [0, 1, 2])
@pytest.mark.parametrize("n", LENGTHS)
def test_axis_length(B, n, axis):
    import torch
    grid = [5, 3, 7]           # ragged tiles beside the long axis
    grid[axis] = n
    grid = tuple(grid)
    p = synth.small_polycrystal(grid, 4, 3)
    rho = np.array([8960.0, 1200.0, 4506.0, 19300.0])
    med = O.Medium(grid, p.L, p.grain_ids, p.C_per_grain, rho)
    k = np.array([[0.31, -0.12, 0.77], [1.0, 0.4, 0.0]]) * math.pi / 1e-3
    u = synth.random_field(grid, 11, batch=2)
    refK = [O.apply_K(med, k[b], u[b]) for b in range(2)]
    refM = [O.apply_M(med, u[b]) for b in range(2)]
    for prec in (0, 1, 2):
        dt = torch.complex64 if prec == 1 else torch.complex128
        plan = B.Plan(grid, p.L, p.grain_ids, p.C_per_grain, rho, B.default_options(precision=min(prec, 1)))
        ud = torch.from_numpy(u).to(device="cuda", dtype=dt).contiguous()
        out = torch.empty_like(ud)
        plan.apply_K(k, ud, out, precision=prec)
        got = out.cpu().numpy()
        for b in range(2):
            assert np.linalg.norm(got[b] - refK[b]) < TOL[prec] * np.linalg.norm(refK[b]), (prec, b)
        if prec == 2:
            continue
        plan.apply_M(ud, out)
        got = out.cpu().numpy()
        for b in range(2):
            assert np.linalg.norm(got[b] - refM[b]) < TOL[prec] * np.linalg.norm(refM[b]), (prec, b)
        plan.apply_K_real(k, ud, out)     # the plain transforms of all three axes
        got = out.cpu().numpy()
        for b in range(2):
            ref = np.fft.ifftn(O.apply_K(med, k[b], np.fft.fftn(u[b], axes=(1, 2, 3))), axes=(1, 2, 3))
            assert np.linalg.norm(got[b] - ref) < TOL[prec] * np.linalg.norm(ref), (prec, b)
        plan.close()
