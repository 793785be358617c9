"""Performance cases of the Bloch-wave library: what its users have it compute.

Each case is one call (or one pair of calls) of the public interface in
`paper_2106_12487_gb300.bloch` on a voxelised periodic cell:

  K       stiffness operator A_k on a batch of Fourier vectors (Plan.apply_K)
  M       mass operator of a two-phase composite, non-uniform density (Plan.apply_M)
  pcg     batched preconditioned CG solves A_k x = b (Plan.pcg)
  props   group velocity and real-space fields with strain of a block of
          eigenvectors (Plan.group_velocity, Plan.eigvec_real)
  bands   band frequencies of a few wave vectors (Plan.solve_bands)

Plans, inputs and output buffers are what a program holds before the call.
Microstructures are periodic Voronoi polycrystals of rotated cubic grains (Cu-like)
and, for M, a long-fibre epoxy/carbon composite.  Vectors have the decaying
spectrum of the solvers' iterates, not white noise.
"""
import math

import numpy as np
import torch

from paper_2106_12487_gb300 import bloch, synth

CELL = 1e-3                       # longest cell edge (m)
PRECISIONS = {"fp32": bloch.FP32, "fp64": bloch.FP64, "ff": bloch.FF}
VOIGT = ((0, 0), (1, 1), (2, 2), (1, 2), (0, 2), (0, 1))


def listed():
    return [
        # One vector on the smallest cell that is solved in earnest (16^3, 8 grains): latency of a single call.
        _K("K_16_fp32_1", 16, 16, 16, 8, 1, "fp32"),
        # A block of ten vectors on the mid-sized cell (64^3, 64 grains, 8 bands + 2 guard vectors).
        _K("K_64_fp32_10", 64, 64, 64, 64, 10, "fp32"),
        # The flagship cell (128^3, 200 grains) with a full subspace block of 18 vectors.
        _K("K_128_fp32_18", 128, 128, 128, 200, 18, "fp32"),
        # The largest cell (256^3, 1000 grains).
        _K("K_256_fp32_2", 256, 256, 256, 1000, 2, "fp32"),
        # A cell whose edges are no powers of two (voxelised measurements, elongated cells).
        _K("K_120x100x84_fp32_6", 120, 100, 84, 100, 6, "fp32"),
        # The plain double-precision form.
        _K("K_64_fp64_4", 64, 64, 64, 64, 4, "fp64"),
        # The float-float operator that checks the converged vectors of the single-precision form.
        _K("K_128_ff_4", 128, 128, 128, 200, 4, "ff"),
        # Mass operator of a long-fibre composite (two densities).
        dict(name="M_128x128x32_fp32_8", op="M", nx=128, ny=128, nz=32, grains=2, nb=8, precision="fp32"),
        # Inner solves of a shift-invert Lanczos step: one system for each of eight wave vectors, loose tolerance.
        dict(name="pcg_128_fp32_8", op="pcg", nx=128, ny=128, nz=128, grains=200, nb=8, precision="fp32", tol=1e-2),
        # Inner solves of the double-precision form, tight tolerance.
        dict(name="pcg_48x40x36_fp64_6", op="pcg", nx=48, ny=40, nz=36, grains=24, nb=6, precision="fp64", tol=1e-10),
        # What follows a band solve: velocities, fields and strains of ten eigenvectors.
        dict(name="props_128_fp32_10", op="props", nx=128, ny=128, nz=128, grains=200, nb=10, precision="fp32"),
        # A whole band solve (single-precision fields, double-precision-class check), two wave vectors.
        dict(name="bands_64_fp32_2x8", op="bands", nx=64, ny=64, nz=64, grains=64, nb=2, bands=8, precision="fp32"),
    ]


def _K(name, nx, ny, nz, grains, nb, precision):
    return dict(name=name, op="K", nx=nx, ny=ny, nz=nz, grains=grains, nb=nb, precision=precision)


def _smooth(lo, hi):
    """Grid sizes the library takes (prime factors 2, 3, 5, 7) in [lo, hi]."""
    out = []
    for n in range(lo, hi + 1):
        m = n
        for p in (2, 3, 5, 7):
            while m % p == 0:
                m //= p
        if m == 1:
            out.append(n)
    return out


def _size(rng, lo, hi):
    """A supported size near a log-uniform one; a power of two two times in five, as users mostly choose."""
    x = math.exp(rng.uniform(math.log(lo), math.log(hi)))
    if rng.random() < 0.4:
        return min(max(2 ** round(math.log2(x)), lo), hi)
    return min(_smooth(lo, hi), key=lambda n: abs(n - x))


# op, precision: weight, edge range, most points (systems x voxels) of a call
_RANGES = [
    ("K", "fp32", 8, (12, 256), 18 * 128 ** 3),
    ("K", "fp64", 2, (12, 128), 2 * 64 ** 3 * 4),
    ("K", "ff", 2, (12, 128), 4 * 128 ** 3),
    ("M", "fp32", 2, (12, 256), 8 * 128 * 128 * 32),
    ("pcg", "fp32", 3, (12, 160), 8 * 128 ** 3),
    ("pcg", "fp64", 1, (12, 48), 6 * 48 * 40 * 36),
    ("props", "fp32", 2, (12, 160), 10 * 128 ** 3),
    ("bands", "fp32", 1, (40, 64), 64 ** 3),
    ("bands", "fp64", 1, (12, 32), 24 ** 3),
]


def draw(rng):
    op, precision, _, (lo, hi), most = rng.choices(_RANGES, weights=[r[2] for r in _RANGES])[0]
    while True:
        if rng.random() < 0.4:                    # a cube
            nx = ny = nz = _size(rng, lo, hi)
        else:
            nx, ny, nz = (_size(rng, lo, hi) for _ in range(3))
        if op in ("K", "M") and rng.random() < 0.1:
            nz = 1                                # a plane cell (cross-section of a long-fibre composite)
        V = nx * ny * nz
        if V <= most:
            break
    if op == "bands":
        return dict(op=op, nx=nx, ny=ny, nz=nz, grains=rng.randint(4, 16), nb=1, bands=rng.randint(3, 6),
                    precision=precision)
    nb = max(1, min(most // V, int(math.exp(rng.uniform(0, math.log(20))))))
    case = dict(op=op, nx=nx, ny=ny, nz=nz, grains=2 if op == "M" else min(200, max(2, V // 4096)), nb=nb,
                precision=precision)
    if op == "pcg":
        case["tol"] = 1e-10 if precision == "fp64" else rng.choice([1e-2, 1e-2, 1e-4])
    return case


# ------------------------------------------------------------------- inputs
def _generator(seed, what):
    return torch.Generator(device="cuda").manual_seed(1000003 * what + seed)


def _lengths(case):
    n = (case["nx"], case["ny"], case["nz"])
    return tuple(CELL * v / max(n) for v in n)


def _cell(case, seed):
    """(grain ids (Nz, Ny, Nx) on the host, stiffness per grain, density per grain)."""
    n = (case["nx"], case["ny"], case["nz"])
    L = _lengths(case)
    if case["op"] == "M":
        frac = 0.4 + 0.2 * ((seed * 7919) % 97) / 97
        p = synth.fibre_composite(n, "circle", frac=frac, n_k=4, L=L)
        return p.grain_ids, p.C_per_grain, p.rho
    G = case["grains"]
    pts = torch.rand(G, 3, generator=_generator(seed, 1), device="cuda", dtype=torch.float64)
    best = torch.full((n[2], n[1], n[0]), math.inf, device="cuda")
    ids = torch.zeros((n[2], n[1], n[0]), device="cuda", dtype=torch.int32)
    d2 = []                                       # squared minimum-image distances per axis, G x N
    for a in range(3):
        x = (torch.arange(n[a], device="cuda", dtype=torch.float64) + 0.5) / n[a]
        d = (x[None, :] - pts[:, a:a + 1]).abs()
        d2.append(((torch.minimum(d, 1 - d) * L[a] / CELL) ** 2).float())
    for g in range(G):
        d = d2[2][g][:, None, None] + d2[1][g][None, :, None] + d2[0][g][None, None, :]
        near = d < best
        best = torch.where(near, d, best)
        ids.masked_fill_(near, g)
    cu = synth.CU_CUBIC
    C6 = synth.cubic_voigt(cu["C11"], cu["C12"], cu["C44"])
    R = synth.haar_rotations(G, 100 + seed)
    C = np.stack([synth.rotate_voigt(C6, R[g]) for g in range(G)])
    return ids.cpu().numpy(), C, np.full(G, cu["rho"])


def _waves(case, seed):
    """nb wave vectors inside the first Brillouin zone, away from its centre."""
    rng = np.random.default_rng(seed)
    L = np.array(_lengths(case))
    return rng.uniform(0.15, 0.95, (case["nb"], 3)) * np.pi / L


def _bins(n):
    m = torch.arange(n, device="cuda", dtype=torch.float64)
    return torch.where(m < (n + 1) // 2, m, m - n)


def _spectrum(case):
    """Amplitude per Fourier bin, 1 / (1 + |m|^2 / 16), m in units of the longest cell edge."""
    L = _lengths(case)
    mx, my, mz = (_bins(case[a]) * (CELL / L[i]) for i, a in enumerate(("nx", "ny", "nz")))
    return 1.0 / (1.0 + (mz[:, None, None] ** 2 + my[None, :, None] ** 2 + mx[None, None, :] ** 2) / 16.0)


def _vectors(case, seed, dtype):
    """nb x 3 x Nz x Ny x Nx Fourier vectors with the decaying spectrum."""
    g = _generator(seed, 2)
    w = _spectrum(case).float()
    out = torch.empty((case["nb"], 3) + tuple(w.shape), device="cuda", dtype=dtype)
    for b in range(case["nb"]):
        for c in range(3):
            re, im = (torch.randn(w.shape, generator=g, device="cuda") for _ in range(2))
            out[b, c] = torch.complex(re * w, im * w)
    return out


def _modes(case, seed, dtype):
    """Fourier vectors whose real-space fields nearly share one phase, as those of eigenvectors do."""
    u = _vectors(case, seed, dtype)
    rng = np.random.default_rng(seed + 5)
    for b in range(case["nb"]):
        turn = complex(np.exp(1j * rng.uniform(-1.2, 1.2)))
        for c in range(3):
            x = torch.fft.ifftn(u[b, c])
            u[b, c] = torch.fft.fftn((x.real + 0.1j * x.imag) * turn)
    return u


def _tensor_type(case):
    return torch.complex64 if case["precision"] == "fp32" else torch.complex128


class State:
    """What a program holds before the call: the plan, the inputs and the buffers for the results."""

    def __init__(self, case, seed):
        self.case = case
        ids, C, rho = _cell(case, seed)
        prec = PRECISIONS[case["precision"]]
        opt = dict(precision=bloch.FP32 if case["precision"] == "fp32" else bloch.FP64)
        if case["op"] == "bands":
            if case["precision"] == "fp32":
                opt.update(method=bloch.LANCZOS, tol_lin=1e-2, tol_eig=1e-5, block=case["bands"] + 2, refine_arith=1)
            else:
                opt.update(method=bloch.LANCZOS, tol_lin=1e-10, tol_eig=1e-10)
        self.plan = bloch.Plan((case["nx"], case["ny"], case["nz"]), _lengths(case), ids, C, rho,
                               bloch.default_options(**opt))
        self.precision = prec
        self.k = _waves(case, seed)
        dt = _tensor_type(case)
        if case["op"] == "bands":
            return
        self.u = _modes(case, seed, dt) if case["op"] == "props" else _vectors(case, seed, dt)
        self.out = torch.empty_like(self.u)
        if case["op"] == "pcg":
            self.u *= synth.CU_CUBIC["rho"]      # the right-hand sides M u of the inverse iteration
        if case["op"] == "props":
            s = list(self.u.shape)
            s[1] = 6
            self.strain = torch.empty(s, device="cuda", dtype=dt)


def prepare(case, seed):
    return State(case, seed)


def run(state):
    case, plan = state.case, state.plan
    op = case["op"]
    if op == "K":
        return plan.apply_K(state.k, state.u, state.out, precision=state.precision)
    if op == "M":
        return plan.apply_M(state.u, state.out)
    if op == "pcg":
        iterations, _, _ = plan.pcg(state.k, state.u, state.out, case["tol"])
        return {"x": state.out, "iterations": iterations}
    if op == "props":
        # the numbers that come back in doubles are as accurate as the vectors given, so they go on in their type
        omega, c = plan.group_velocity(state.k, state.u)
        phi = plan.eigvec_real(state.u, state.out, state.strain)
        return {"omega": omega.astype(np.float32), "c": c.astype(np.float32), "phi": phi.astype(np.float32),
                "u": state.out, "strain": state.strain}
    omega, _, status = plan.solve_bands(state.k, case["bands"])
    return {"omega": omega, "status": status}


# --------------------------------------------------------------------- work
def work(case):
    """Least memory traffic and arithmetic of one pass.

    One operator: input, output and grain ids once; 36 one-dimensional
    transforms per voxel (six strain components in, six stress components out,
    along three axes) at 5 log2 N operations a point, strain 24, stress 144,
    divergence 30.  A solve counts what its iterations cannot do without, for
    about as many iterations as these cells need.
    """
    V = case["nx"] * case["ny"] * case["nz"]
    nb, size = case["nb"], 8 if case["precision"] == "fp32" else 16
    logs = sum(math.log2(case[a]) for a in ("nx", "ny", "nz"))
    field = 3 * V * size
    apply_flops = V * (12 * 5 * logs + 198)
    op = case["op"]
    if op == "K":
        return {"bytes": nb * 2 * field + 4 * V, "flops": nb * apply_flops}
    if op == "M":
        return {"bytes": nb * 2 * field + 4 * V, "flops": nb * V * (6 * 5 * logs + 6)}
    if op == "pcg":
        its = 4 if case["tol"] >= 1e-2 else 8 if case["tol"] >= 1e-4 else 20
        # x, r and p are read and written each iteration
        return {"bytes": nb * its * 6 * field, "flops": nb * its * (apply_flops + V * 120)}
    if op == "props":
        return {"bytes": nb * (4 * field + 2 * field), "flops": nb * V * (12 * 5 * logs + 168 + 120 + 9 * 5 * logs + 60)}
    # about 60 operator applies per eigenpair in the single-precision form, 400 in the double-precision one
    applies = case["nb"] * case["bands"] * (60 if case["precision"] == "fp32" else 400)
    return {"bytes": applies * 4 * field, "flops": applies * apply_flops}


# -------------------------------------------------------------------- exact
class _Exact:
    """The operators in 64 bits with torch FFTs, one vector at a time."""

    def __init__(self, case, seed):
        self.n = (case["nx"], case["ny"], case["nz"])
        ids, C, rho = _cell(case, seed)
        self.ids = torch.from_numpy(np.ascontiguousarray(ids)).cuda().long()
        self.C = torch.from_numpy(C).cuda()
        self.rho = torch.from_numpy(rho).cuda()
        L = _lengths(case)
        self.xi = [2 * math.pi / L[a] * _bins(self.n[a]) for a in range(3)]
        share = torch.bincount(self.ids.reshape(-1), minlength=len(rho)).double() / self.ids.numel()
        self.C0 = (share[:, None, None] * self.C).sum(0)

    def q(self, k):
        x, y, z = (self.xi[a] + float(k[a]) for a in range(3))
        return [x[None, None, :], y[None, :, None], z[:, None, None]]

    def stress(self, k, u):
        """Fourier transform of C : sym((xi + k) (x) u), Voigt order."""
        q = self.q(k)
        eps = []
        for i, j in VOIGT:
            e = q[i] * u[i] if i == j else q[i] * u[j] + q[j] * u[i]
            eps.append(torch.fft.ifftn(e))
        out = []
        for a in range(6):
            s = torch.zeros_like(eps[0])
            for b in range(6):
                s += self.C[:, a, b][self.ids] * eps[b]
            out.append(torch.fft.fftn(s))
        return out

    @staticmethod
    def divergence(q, s):
        return torch.stack([q[0] * s[0] + q[1] * s[5] + q[2] * s[4], q[0] * s[5] + q[1] * s[1] + q[2] * s[3],
                            q[0] * s[4] + q[1] * s[3] + q[2] * s[2]])

    def K(self, k, u):
        return self.divergence(self.q(k), self.stress(k, u))

    def M(self, u):
        return torch.stack([torch.fft.fftn(self.rho[self.ids] * torch.fft.ifftn(c)) for c in u])

    def green(self, k):
        """The inverse of P_ik = C0_ijkl q_j q_l at every Fourier voxel."""
        V6 = {}
        for a, (i, j) in enumerate(VOIGT):
            V6[i, j] = V6[j, i] = a
        q = self.q(k)
        P = torch.zeros((self.n[2], self.n[1], self.n[0], 3, 3), device="cuda", dtype=torch.float64)
        for i in range(3):
            for m in range(3):
                for j in range(3):
                    for l in range(3):
                        P[..., i, m] += self.C0[V6[i, j], V6[m, l]] * q[j] * q[l]
        return torch.linalg.inv(P)

    def pcg(self, k, b, tol):
        Z = self.green(k)

        def precond(r):
            return torch.stack([sum(Z[..., i, j] * r[j] for j in range(3)) for i in range(3)])

        def dot(a, c):
            return torch.vdot(a.reshape(-1), c.reshape(-1)).real
        x, r = torch.zeros_like(b), b.clone()
        p = z = precond(r)
        rz, bb, its = dot(r, z), dot(b, b), 0
        while dot(r, r) > tol * tol * bb and its < 10000:
            Ap = self.K(k, p)
            alpha = rz / dot(p, Ap)
            x += alpha * p
            r -= alpha * Ap
            z = precond(r)
            new = dot(r, z)
            p = z + (new / rz) * p
            rz = new
            its += 1
        return x, its


def exact(case, seed):
    op = case["op"]
    if op == "bands":
        return None
    E = _Exact(case, seed)
    k = _waves(case, seed)
    dt = _tensor_type(case)
    u = _modes(case, seed, dt) if op == "props" else _vectors(case, seed, dt)
    nb = case["nb"]
    out = torch.empty(u.shape, device="cuda", dtype=torch.complex128)
    if op in ("K", "M"):
        for b in range(nb):
            v = u[b].to(torch.complex128)
            out[b] = E.K(k[b], v) if op == "K" else E.M(v)
        return out
    if op == "pcg":
        u *= synth.CU_CUBIC["rho"]
        its = []
        for b in range(nb):
            out[b], n = E.pcg(k[b], u[b].to(torch.complex128), case["tol"])
            its.append(n)
        return {"x": out, "iterations": np.array(its, dtype=np.int32)}
    strain = torch.empty((nb, 6) + tuple(u.shape[2:]), device="cuda", dtype=torch.complex128)
    omega, c, phi = np.zeros(nb), np.zeros((nb, 3)), np.zeros(nb)
    index = ((0, 5, 4), (5, 1, 3), (4, 3, 2))
    xi = [E.xi[0][None, None, :], E.xi[1][None, :, None], E.xi[2][:, None, None]]
    for b in range(nb):
        v = u[b].to(torch.complex128)
        S = E.stress(k[b], v)
        Kv = E.divergence(E.q(k[b]), S)
        uMu = float(torch.vdot(v.reshape(-1), E.M(v).reshape(-1)).real)
        lam = float(torch.vdot(v.reshape(-1), Kv.reshape(-1)).real) / uMu
        omega[b] = math.sqrt(lam)
        for m in range(3):
            d = sum(float(torch.vdot(v[i].reshape(-1), S[index[i][m]].reshape(-1)).real) for i in range(3))
            c[b, m] = 2 * d / uMu / (2 * omega[b])
        x = torch.stack([torch.fft.ifftn(w) for w in v])
        s = complex((x * x).sum())
        phi[b] = 0.5 * math.atan2(s.imag, s.real)
        turn = complex(math.cos(phi[b]), -math.sin(phi[b]))
        out[b] = turn * x
        for a, (i, j) in enumerate(VOIGT):
            strain[b, a] = turn * torch.fft.ifftn(0.5j * (xi[j] * v[i] + xi[i] * v[j]))
    return {"omega": omega, "c": c, "phi": phi, "u": out, "strain": strain}
