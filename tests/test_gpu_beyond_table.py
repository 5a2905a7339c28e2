"""The float x pass's recovery of voxels whose overstress lies beyond the direct rate tables
(mc_recover with the strain path in shared memory), in the trial passes and the commit: a full
solve against the oracle, alone and in a group.  The tables of this law end at 41 MPa (slip) and
0.04 MPa (twins); 45 lines of 6 voxels leave the last CTA partly empty."""
import dataclasses

import numpy as np
import pytest

from helpers import six_to_tensor
from oracle import rve_oracle as orc

pytestmark = pytest.mark.gpu

LAW = dict(K=0.01, Kt=1e-5)


def test_float_solve_beyond_the_tables(lib, cuda):
    from paper_2402_09996_gb300 import rve

    rng = np.random.default_rng(12)
    gid = rng.integers(0, 4, size=(5, 9, 6)).astype(np.uint32)
    gid.flat[:4] = [0, 1, 2, 3]
    euler = rng.uniform(0.0, 1.5, size=(4, 3))

    def make(**kw):
        s = rve.RVE(gid, euler, precision=rve.FP32, fixed_iters=6, **kw)
        s.set_material(**LAW)
        s.set_mixed_load(dt=0.5)
        return s

    with make() as s:
        s.step(5)
        got, sig, v = s.history(), s.field(rve.FIELD_STRESS), s.field(rve.FIELD_V)
    ref = orc.OracleRVE(gid.astype(np.int64), euler, dataclasses.replace(orc.Material(), **LAW),
                        orc.Options(fixed_iters=6))
    ref.set_load(orc.Load(dt=0.5))
    ref.run(5)
    # inside the twins' table the slip of 2.5 s stays below 2.5 * 0.04 / eta = 1e-5
    assert v.reshape(16, -1)[12:].max() > 1e-5
    # the bounds of the other FP32 solves
    for g, r in zip(got, ref.history):
        assert np.max(np.abs(g["S"] - r["S"])) < 1e-4 * np.max(np.abs(r["S"]))
        assert abs(g["mean_v"] - r["mean_v"]) <= 1e-4 * abs(r["mean_v"]) + 1e-12
        assert abs(g["mean_f"] - r["mean_f"]) <= 1e-4 * abs(r["mean_f"]) + 1e-12
    sig_ref = ref.fields()["sigma"]
    assert np.linalg.norm(six_to_tensor(sig) - sig_ref) < 1e-3 * np.linalg.norm(sig_ref)
    pair = [make(batch_group=True), make(batch_group=True)]
    try:
        rve.step_batch(pair, 5)
        for s in pair:
            assert np.array_equal(s.field(rve.FIELD_STRESS), sig) and np.array_equal(s.field(rve.FIELD_V), v)
    finally:
        for s in pair:
            s.close()
