"""Digits of the doubles that the band properties return for FP32 vectors: the
products of FP32 values are formed exactly and summed to about 48 bits, so
nothing is lost beside the fields' own FP32 roundings."""
import numpy as np
import pytest

from paper_2106_12487_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def B():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2106_12487_gb300 import bloch, build
    build.build()
    bloch.lib()
    return bloch


def to_dev(a):
    import torch
    return torch.from_numpy(np.ascontiguousarray(a)).to(device="cuda", dtype=torch.complex64)


@pytest.mark.parametrize("rho_mix", [False, True])
def test_frequency_and_velocity_where_the_stress_is_exact(B, rho_mix):
    """Homogeneous cell of 4^3 points (its transforms need no roundings for a
    constant field), one coefficient in bin 0, polarisation y, q along x: the
    stress is c44 q u with q and c44 short binary fractions, exact in FP32 for
    20-bit u, and omega = q sqrt(c44 / rho), d omega / d k = sqrt(c44 / rho) e_x
    with the mean density rho, for every u. Sums of 48 bits: 1e-13 leaves an order of
    magnitude."""
    L = 2.0 * np.pi                       # scaled wave numbers equal the unscaled ones
    C = np.diag([1.0, 1.0, 1.0, 0.375, 0.375, 0.375])
    rng = np.random.default_rng(5)
    nb = 16
    ids = np.arange(64, dtype=np.int32) % 2
    rho = np.array([1.0, 3.0]) if rho_mix else np.array([2.0, 2.0])   # mean 2; M u is exact too
    plan = B.Plan((4, 4, 4), (L, L, L), ids, np.stack([C, C]), rho, B.default_options(precision=1))
    u = np.zeros((nb, 3, 4, 4, 4), dtype=complex)
    u[:, 1, 0, 0, 0] = (rng.integers(1 << 19, 1 << 20, nb) + 1j * rng.integers(1 << 19, 1 << 20, nb)) * 2.0 ** -20
    k = np.tile([0.5, 0.0, 0.0], (nb, 1))
    om, c = plan.group_velocity(k, to_dev(u))
    v = np.sqrt(0.375 / 2)
    assert np.max(np.abs(om / (0.5 * v) - 1)) < 1e-13
    assert np.max(np.abs(c[:, 0] / v - 1)) < 1e-13 and np.max(np.abs(c[:, 1:])) == 0


@pytest.mark.parametrize("grid", [(12, 10, 8), (9, 7, 5), (32, 16, 16)])
def test_phase_of_fp32_vectors(B, grid):
    """phi = arg(sum_m U(m) U(-m)) / 2 of the FP32 values in FP64.  The sum of
    the absolute terms is about the sum here (vectors of one phase, perturbed by
    a tenth), so 48-bit sums give phi to a few 1e-15; 1e-12 leaves room for it."""
    import torch
    rng = np.random.default_rng(8)
    nb = 5
    shape = (nb, 3) + tuple(reversed(grid))
    real = rng.normal(size=shape)
    pert = rng.normal(size=shape) + 1j * rng.normal(size=shape)
    w = np.exp(1j * rng.uniform(-1.4, 1.4, nb))[:, None, None, None, None] * real + 0.1 * pert
    U = np.fft.fftn(w, axes=(2, 3, 4)).astype(np.complex64)
    plan = B.Plan.from_problem(synth.small_polycrystal(grid, 5, 17), precision=1)
    d = to_dev(U)
    phi = plan.eigvec_real(d, torch.empty_like(d), None)
    V = U.astype(np.complex128)
    mirror = V
    for ax in (2, 3, 4):
        mirror = np.roll(np.flip(mirror, ax), 1, ax)
    want = 0.5 * np.angle((V * mirror).reshape(nb, -1).sum(1))
    assert np.max(np.abs(np.exp(2j * phi) - np.exp(2j * want))) < 1e-12
