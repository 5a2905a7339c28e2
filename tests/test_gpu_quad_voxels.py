"""The FP64 x pass with four lanes per voxel (mc_voxel_quad) against the oracle: lines and CTAs
that leave warps and turns partly empty, a table for each law, and a material set afterwards
whose exponents have no direct table (one lane per voxel)."""
import dataclasses

import numpy as np
import pytest

from oracle.rve_oracle import Material, OracleRVE, Options

pytestmark = pytest.mark.gpu

LAWS = {"workload": {}, "two_tables": dict(n=6.42, nt=4.0, K=104.0, Kt=60.0), "no_table": dict(n=12.0, nt=11.0)}


@pytest.mark.parametrize("shape,law", [((2, 3, 2), "workload"), ((5, 9, 6), "workload"), ((4, 15, 10), "two_tables"),
                                       ((8, 12, 18), "workload"), ((5, 9, 6), "no_table")])
def test_small_fp64_grids_match_oracle(lib, cuda, shape, law):
    from paper_2402_09996_gb300 import rve

    rng = np.random.default_rng(sum(shape))
    gid = rng.integers(0, 3, size=shape).astype(np.uint32)
    gid.flat[:3] = [0, 1, 2]
    euler = rng.uniform(0.0, 1.5, size=(3, 3))
    with rve.RVE(gid, euler, precision=rve.FP64, fixed_iters=4) as s:
        if LAWS[law]:
            s.set_material(**LAWS[law])
        s.step(3)
        got, v = s.history(), s.field(rve.FIELD_V)
    ref = OracleRVE(gid.astype(np.int64), euler, dataclasses.replace(Material(), **LAWS[law]), Options(fixed_iters=4))
    ref.run(3)
    for g, r in zip(got, ref.history):
        assert np.max(np.abs(g["S"] - r["S"])) < 1e-9 * np.max(np.abs(r["S"]))
        assert abs(g["mean_v"] - r["mean_v"]) <= 1e-9 * abs(r["mean_v"]) + 1e-15
    assert np.any(v > 0)
