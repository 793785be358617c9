"""FP32 conjugate gradients over the range of their numbers."""
import math

import numpy as np
import pytest

from paper_2106_12487_gb300 import synth

pytestmark = pytest.mark.gpu
GRIDS = [(12, 10, 8), (32, 16, 64)]   # mixed-radix and two-stage passes


@pytest.fixture(scope="module")
def B():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2106_12487_gb300 import bloch, build
    build.build()
    bloch.lib()
    return bloch


def solve(B, plan, k, b, tol, max_iter=500, x0=None):
    import torch
    bd = torch.from_numpy(b).to(device="cuda", dtype=torch.complex64).contiguous()
    x = torch.empty_like(bd) if x0 is None else torch.from_numpy(x0).to(device="cuda", dtype=torch.complex64).contiguous()
    iters, rel, st = plan.pcg(k, bd, x, tol, max_iter, x0=x0 is not None, allow_nonconv=True)
    return x.cpu().numpy(), iters, rel, st


@pytest.mark.parametrize("amp", [1e3, 1e4, 1e8])
@pytest.mark.parametrize("grid", GRIDS)
def test_large_irreducible_part(B, grid, amp):
    """k = 0 with bin 0 far above the rest: (r, r) stays at its square while
    (r, z) falls by 32 digits, so a scale that fits one does not fit the other."""
    plan = B.Plan.from_problem(synth.small_polycrystal(grid, 5, 7), precision=1)
    k = np.zeros((1, 3))
    b = synth.random_field(grid, 3, batch=1) * 1e18
    b[..., 0, 0, 0] = 0
    want, _, _, st = solve(B, plan, k, b, 1e-6)
    assert st == 0
    b[..., 0, 0, 0] = amp * np.abs(b).max()
    x, iters, rel, st = solve(B, plan, k, b, 1e-6, 2000)
    assert st == 4 and iters[0] < 1000 and np.isfinite(x).all()
    # what is left of r is bin 0: its share of ||b||, to FP32 sums
    assert abs(rel[0] - np.linalg.norm(b[..., 0, 0, 0]) / np.linalg.norm(b)) < 1e-5
    # same bound as for amplitude 1: a small condition number times the tolerance
    assert np.linalg.norm(x - want) < 1e-4 * np.linalg.norm(want)


@pytest.mark.parametrize("use_x0", [False, True])
@pytest.mark.parametrize("e", [-75, -60, 40, 64])
@pytest.mark.parametrize("grid", GRIDS)
def test_right_hand_sides_of_any_size(B, grid, e, use_x0):
    """A power of two on b (and x0) changes no digit of a step, so iterations
    and solution are those of b, also where the squares of b over the operator's
    scale (about 7e18 here) leave the FP32 range."""
    plan = B.Plan.from_problem(synth.small_polycrystal(grid, 5, 7), precision=1)
    k = np.array([[0.4, 0.2, -0.3], [0.9, 0.0, 0.1]]) * math.pi / 1e-3
    b = (synth.random_field(grid, 3, batch=2) * 1e18).astype(np.complex64)
    x0 = solve(B, plan, k, b, 1e-1)[0] if use_x0 else None
    f = np.float32(2.0 ** e)
    ref, it0, rel0, st0 = solve(B, plan, k, b, 1e-5, x0=x0)
    x, it, rel, st = solve(B, plan, k, b * f, 1e-5, x0=None if x0 is None else x0 * f)
    assert st0 == 0 and st == 0 and np.array_equal(it, it0) and it.min() > 0
    assert np.allclose(rel, rel0, rtol=1e-5)
    assert np.linalg.norm(x.astype(np.complex128) * 2.0 ** -e - ref) <= 1e-6 * np.linalg.norm(ref)


@pytest.mark.parametrize("grid", GRIDS)
def test_tolerance_below_the_fp32_digits(B, grid):
    """The recursive residual of a system that can converge is followed as far
    as asked, and a tolerance that is not reached within the cap takes the
    iterations of the cap."""
    plan = B.Plan.from_problem(synth.small_polycrystal(grid, 5, 7), precision=1)
    k = np.array([[0.4, 0.2, -0.3]]) * math.pi / 1e-3
    b = synth.random_field(grid, 3, batch=1) * 1e18
    _, iters, rel, st = solve(B, plan, k, b, 1e-20)
    assert st == 0 and rel[0] <= 1e-20 and iters[0] < 500
    _, n, _, st = solve(B, plan, k, b, 1e-30, max_iter=int(iters[0]) - 1)
    assert st == 4 and n[0] == iters[0] - 1
