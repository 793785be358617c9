"""BLOCH_LOBPCG converges whatever the last bit: wave vectors that differ by
1e-7 of each other, cells of several seeds and sizes, uniform and per-grain
densities, near and far from Gamma; frequencies against the shift-invert
Lanczos form in FP64."""
import dataclasses
import math

import numpy as np
import pytest

from paper_2106_12487_gb300 import synth

pytestmark = pytest.mark.gpu
# relative frequency error at the stop tests' residuals, as test_lobpcg_matches_oracle
FORMS = {"fp64": (1e-9, dict(precision=0, tol_lin=1e-10, tol_eig=1e-10)),
         "fp32": (1e-6, dict(precision=1, tol_lin=1e-3, tol_eig=1e-5))}


@pytest.fixture(scope="module")
def B():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2106_12487_gb300 import bloch, build
    build.build()
    bloch.lib()
    return bloch


def cell(grid, grains, seed, rho_mix):
    p = synth.small_polycrystal(grid, grains, seed)
    if rho_mix:
        p = dataclasses.replace(p, rho=np.random.default_rng(8).uniform(3000.0, 9000.0, p.G))
    return p


def lobpcg(B, p, ks, n, opt):
    plan = B.Plan.from_problem(p, method=B.LOBPCG, max_outer=100, **opt)
    got, stats, st = plan.solve_bands(ks, n, allow_nonconv=True)
    plan.close()
    assert st == 0, stats
    return got


def lanczos(B, p, ks, n):
    plan = B.Plan.from_problem(p, method=B.LANCZOS, precision=0, tol_lin=1e-11, tol_eig=1e-10)
    want = plan.solve_bands(ks, n)[0]
    plan.close()
    return want


@pytest.mark.parametrize("form", list(FORMS))
@pytest.mark.parametrize("rho_mix", [False, True])
def test_neighbouring_wave_vectors(B, form, rho_mix):
    bar, opt = FORMS[form]
    path = np.array([[0.0, 0.0, 0.0], [0.15, 0.0, 0.0], [0.6, 0.3, 0.0]]) * math.pi / 1e-3
    for seed in (19, 20, 21):
        p = cell((12, 10, 8), 6, seed, rho_mix)
        for e in (0.0, 1e-7, 2e-7, 5e-7, 1e-6, 3e-6):
            got = lobpcg(B, p, path * (1 + e), 6, opt)
            if e == 0.0:
                want = lanczos(B, p, path, 6)
                assert np.max(np.abs(got - want)) <= bar * np.max(want)
                assert np.max(np.abs(got[1:] / want[1:] - 1)) <= bar


@pytest.mark.parametrize("form", list(FORMS))
@pytest.mark.parametrize("grid,grains", [((24, 24, 24), 12), ((40, 36, 30), 20), ((64, 64, 64), 64)])
def test_larger_cells(B, form, grid, grains):
    if form == "fp64" and grid[0] > 40:
        pytest.skip("covered by the smaller cells")
    bar, opt = FORMS[form]
    ks = np.array([[0.6, 0.3, 0.0], [0.37, 0.21, -0.29], [0.05, 0.02, 0.0]]) * math.pi / 1e-3
    for rho_mix in (False, True):
        p = cell(grid, grains, 5, rho_mix)
        want = lanczos(B, p, ks, 8)
        for i in range(len(ks)):
            got = lobpcg(B, p, ks[i:i + 1], 8, opt)
            assert np.max(np.abs(got[0] / want[i] - 1)) <= bar
