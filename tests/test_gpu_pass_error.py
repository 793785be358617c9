"""The plan's pass error word (a staging wait that ran out) is reported by the
synchronising call whose passes set it.  The word is set by a copy from a small
helper built against the plan's declaration: no wait is made to run out."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

from paper_2106_12487_gb300 import synth

pytestmark = pytest.mark.gpu
GRID = (16, 16, 32)

HELPER = r"""
#include "internal.h"
extern "C" int raise_pass_error(void* plan) {
    const int one = 1;
    return (int)cudaMemcpy(((bloch_plan*)plan)->d_perr, &one, sizeof(int), cudaMemcpyHostToDevice);
}
"""


@pytest.fixture(scope="module")
def B():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2106_12487_gb300 import bloch, build
    build.build()
    bloch.lib()
    return bloch


@pytest.fixture(scope="module")
def raise_error(tmp_path_factory):
    from paper_2106_12487_gb300 import build
    d = tmp_path_factory.mktemp("helper")
    src, lib = os.path.join(d, "raise.cu"), os.path.join(d, "libraise.so")
    with open(src, "w") as f:
        f.write(HELPER)
    subprocess.run([build.nvcc(), "-shared", *build.ARCH, *build.FLAGS, "-o", lib, src], check=True)
    fn = ctypes.CDLL(lib).raise_pass_error
    fn.argtypes = [ctypes.c_void_p]
    return fn


@pytest.mark.parametrize("call", ["group_velocity", "eigvec_real", "pcg", "solve_bands"])
def test_the_call_reports_it_once(B, raise_error, call):
    import torch
    plan = B.Plan.from_problem(synth.small_polycrystal(GRID, 5, 17), precision=1)
    k = np.array([[500.0, 200.0, -300.0]])
    u = torch.from_numpy(synth.random_field(GRID, 3, batch=1).astype(np.complex64)).cuda()
    out = torch.empty_like(u)
    calls = {"group_velocity": lambda: plan.group_velocity(k, u),
             "eigvec_real": lambda: plan.eigvec_real(u, out),
             "pcg": lambda: plan.pcg(k, u, out, 1e-3),
             "solve_bands": lambda: plan.solve_bands(k, 2, allow_nonconv=True)}
    calls[call]()
    torch.cuda.synchronize()
    assert raise_error(plan.handle) == 0
    with pytest.raises(B.BlochError) as e:
        calls[call]()
    assert "ECUDA" in str(e.value)
    calls[call]()          # reported once, then cleared
