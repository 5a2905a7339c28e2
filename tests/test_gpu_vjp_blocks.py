"""The reverse pass of increments with more than 4 substeps (adjoint.cuh, blocks of kBlockVjp):
its device memory, and its gradients at whole and ragged block counts."""
import os
import subprocess
import sys
from pathlib import Path

import numpy as np
import pytest

from oracle import rve_oracle as orc
from test_gpu_adjoint import _history_J
from test_gpu_vjp_records import test_reverse_pass_matches_finite_differences as _check_points

pytestmark = pytest.mark.gpu

# Device memory that the context takes for a call with 1 substep and then for one with nsub.
_MEMORY = """
import sys, torch
from paper_2402_09996_gb300 import rve
torch.zeros(1, device="cuda")
def free():
    torch.cuda.synchronize()
    return torch.cuda.mem_get_info()[0]
z = lambda k: torch.zeros((k, 64), device="cuda", dtype=torch.float64)
R = torch.eye(3, device="cuda", dtype=torch.float64).reshape(1, 9).repeat(64, 1)
e = z(6)
before = free()
rve.material_point_vjp(R, e, e, z(34), z(6), z(34), 0.125 * int(sys.argv[1]), int(sys.argv[1]), rve.FP64)
print(before - free(), torch.cuda.get_device_properties(0).multi_processor_count)
"""


@pytest.mark.parametrize("nsub", [8, 16])
def test_reservation_of_long_increments(lib, cuda, nsub):
    """CUDA reserves a kernel's local memory for 2048 threads an SM.  The kernels kept 24.4 KB a
    thread before records were stored, so a call that fitted then takes no more than that now."""
    root = Path(__file__).resolve().parent.parent
    out = subprocess.run([sys.executable, "-c", _MEMORY, str(nsub)], cwd=root, env={**os.environ, "PYTHONPATH": str(root)},
                         check=True, capture_output=True, text=True).stdout.split()
    assert int(out[0]) <= 24432 * 2048 * int(out[1]), out


@pytest.mark.parametrize("n,nsub", [(33, 8), (33, 9), (65, 13)])
def test_points_over_several_blocks(lib, cuda, n, nsub):
    _check_points(lib, cuda, n, nsub, {})


@pytest.mark.parametrize("nsub", [8, 9])
def test_history_gradient_over_several_blocks(lib, cuda, nsub):
    """The tangent's seven sweeps per block, against central differences of the forward solve (bounds
    of test_gpu_adjoint.py)."""
    from oracle.voronoi import label_rve

    from paper_2402_09996_gb300 import inputs, rve

    inp = inputs.make_inputs((8, 6, 10), 3, 0.5, seed=17)
    gid = label_rve(inp)
    n_inc, dt = 3, 0.5
    opts = dict(tol=1e-12, max_iter=3000, n_sub=nsub)
    _, S0 = _history_J(gid, inp.euler, {}, np.zeros(n_inc), n_inc, dt, **opts)
    target = 0.97 * S0
    J, gp, _, _ = rve.history_gradient(gid, inp.euler, n_inc, dt, target, **opts)
    for name in ("r0_ord", "Q_s", "c"):
        k = rve.PARAM_NAMES.index(name)
        p0 = getattr(orc.Material(), name)
        h = 1e-5 * abs(p0)
        num = (_history_J(gid, inp.euler, {name: p0 + h}, target, n_inc, dt, **opts)[0] -
               _history_J(gid, inp.euler, {name: p0 - h}, target, n_inc, dt, **opts)[0]) / (2 * h)
        assert abs(num - gp[k]) <= 1e-4 * max(abs(num), abs(gp[k])) + 1e-9 * J / abs(p0), (name, num, gp[k])
