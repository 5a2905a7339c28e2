"""The direct tables of the regularised rate (rate_table.cuh) against the FP64 oracle: laws at
the edges of the tabulated exponents, slip and twin laws with a table each, arguments below
and beyond the table, and exponents outside the tabulated range."""
import dataclasses

import numpy as np
import pytest

from helpers import rel_err, six_to_tensor, tensor_to_six
from oracle import rve_oracle as orc
from test_gpu_kernels import _random_material_points

pytestmark = pytest.mark.gpu

LAWS = {
    "largest_n_and_smallest_nt": dict(n=10.2, nt=2.0, K=10.0, Kt=50.0),
    "coarse_segments": dict(n=2.5, nt=5.0, K=100.0, Kt=100.0),
    # the table ends at 0.04 .. 41 MPa: most overstresses lie beyond it
    "beyond_the_table": dict(K=0.01, Kt=1e-5),
    "no_table": dict(n=12.0, nt=1.5),
    # a saturated twin fraction (prefactor 0) and rates far below the table's floor
    "no_twin_left": dict(fm=1e-4, n=10.0, nt=10.0),
}


@pytest.mark.parametrize("prec", ["fp64", "fp32"])
@pytest.mark.parametrize("law", list(LAWS))
@pytest.mark.parametrize("n", [33])
def test_tabulated_rates_match_oracle(lib, cuda, law, prec, n):
    import torch

    from paper_2402_09996_gb300 import rve

    p = rve.FP64 if prec == "fp64" else rve.FP32
    tdt = torch.float64 if p == rve.FP64 else torch.float32
    R, eps_n, eps, ep, v, al = _random_material_points(n, 91)
    if p == rve.FP32:
        R, eps_n, eps, ep, v, al = (a.astype(np.float32).astype(np.float64) for a in (R, eps_n, eps, ep, v, al))
    dt = 0.5
    nsub = orc.default_n_sub(dt)
    mat = dataclasses.replace(orc.Material(), **LAWS[law])
    sig_ref, ep_ref, v_ref, al_ref = orc.material_point_increment(mat, R, eps_n, eps, ep, v, al, dt, nsub)
    to_dev = lambda a: torch.tensor(np.ascontiguousarray(a), device=cuda, dtype=tdt)  # noqa: E731
    st = to_dev(np.concatenate([tensor_to_six(ep), v.T, al.T], axis=0))
    sig = rve.material_point(to_dev(R.reshape(n, 9)), to_dev(tensor_to_six(eps_n)), to_dev(tensor_to_six(eps)), st,
                             dt, nsub, p, **LAWS[law]).cpu().numpy()
    st = st.cpu().numpy()
    tol = 1e-10 if p == rve.FP64 else 2e-4  # the bounds of the other material-point comparisons
    assert rel_err(six_to_tensor(sig), sig_ref) < tol
    assert rel_err(six_to_tensor(st[:6]), ep_ref) < tol
    assert rel_err(st[6:22].T, v_ref) < tol
    assert rel_err(st[22:].T, al_ref) < tol
    assert 0.05 < np.any(np.abs(v_ref - v) > 0, axis=1).mean() < 0.999
