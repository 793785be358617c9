"""Conjugate gradients whose residual update is fused into the divergence pass:
independence of the size of the right-hand side in FP32, and the stop of a
system whose remaining residual no step can reduce (bin 0 at k = 0)."""
import math

import numpy as np
import pytest

from paper_2106_12487_gb300 import synth

pytestmark = pytest.mark.gpu
GRIDS = [(12, 10, 8), (32, 16, 64), (64, 9, 16), (256, 4, 6)]   # mixed-radix and two-stage passes


@pytest.fixture(scope="module")
def B():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2106_12487_gb300 import bloch, build
    build.build()
    bloch.lib()
    return bloch


def solve(B, plan, k, b, prec, tol, max_iter=500):
    import torch
    bd = torch.from_numpy(b).to(device="cuda", dtype=torch.complex64 if prec else torch.complex128).contiguous()
    x = torch.empty_like(bd)
    iters, _, st = plan.pcg(k, bd, x, tol, max_iter, allow_nonconv=True)
    return x.cpu().numpy(), iters, st


@pytest.mark.parametrize("grid", GRIDS)
def test_pcg_fp32_scales_with_its_right_hand_side(B, grid):
    """Scaling b by a power of two scales every step exactly: same iterations,
    same digits."""
    p = synth.small_polycrystal(grid, 5, 7)
    plan = B.Plan.from_problem(p, precision=1)
    k = np.array([[0.4, 0.2, -0.3], [0.9, 0.0, 0.1]]) * math.pi / 1e-3
    b = (synth.random_field(grid, 3, batch=2) * 1e18).astype(np.complex64)
    x0, it0, st0 = solve(B, plan, k, b, 1, 1e-5)
    assert st0 == 0
    for e in (-44, 24):
        x, it, st = solve(B, plan, k, b * np.float32(2.0 ** e), 1, 1e-5)
        assert st == 0 and np.array_equal(it, it0)
        assert np.linalg.norm(x * 2.0 ** -e - x0) <= 1e-6 * np.linalg.norm(x0)


@pytest.mark.parametrize("prec", [0, 1])
@pytest.mark.parametrize("grid", GRIDS[:3])
def test_pcg_ends_on_an_irreducible_residual(B, grid, prec):
    """k = 0 with a right-hand side in bin 0: reported as not converged, well
    before the cap, with the solution of the rest (error at most a small
    condition number times the tolerance)."""
    p = synth.small_polycrystal(grid, 5, 7)
    plan = B.Plan.from_problem(p, precision=prec)
    k = np.zeros((1, 3))
    b = synth.random_field(grid, 3, batch=1) * 1e18
    b[..., 0, 0, 0] = 0
    want, _, st = solve(B, plan, k, b, prec, 1e-6)
    assert st == 0
    b[..., 0, 0, 0] = np.abs(b).max()
    x, iters, st = solve(B, plan, k, b, prec, 1e-6, 2000)
    assert st == 4 and iters[0] < 1000 and np.isfinite(x).all()
    assert np.linalg.norm(x - want) < 1e-4 * np.linalg.norm(want)
