"""The reverse pass's stage records (adjoint.cuh, VjpStage) at the edges of their ranges: one
substep, the largest count of the small variant and one more, the largest count; a single
point, one warp and a point, several blocks.  Directional derivatives against central
differences of the FP64 oracle, with the bounds of test_gpu_adjoint.py."""
import dataclasses

import numpy as np
import pytest

from oracle import rve_oracle as orc
from test_gpu_adjoint import PARAMS, _J, _points

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,nsub,law", [(1, 4, {}), (33, 1, {}), (33, 5, {}), (65, 16, {}), (129, 4, {}),
                                        (33, 4, dict(n=12.0, nt=11.0))])
def test_reverse_pass_matches_finite_differences(lib, cuda, n, nsub, law):
    import torch

    from paper_2402_09996_gb300 import rve

    dt = 0.125 * nsub
    mat = dataclasses.replace(orc.Material(), **law)
    R, en6, e6, ep6, v, al = _points(n, 40 + n + nsub, 1.0)
    rng = np.random.default_rng(7)
    sb, yb = rng.normal(size=(6, n)) * 1e-2, rng.normal(size=(34, n)) * 10.0
    to = lambda a: torch.tensor(np.ascontiguousarray(a), device=cuda, dtype=torch.float64)  # noqa: E731
    st_b = to(yb)
    out = rve.material_point_vjp(to(R.reshape(n, 9)), to(en6), to(e6), to(np.concatenate([ep6, v.T, al.T], axis=0)),
                                 to(sb), st_b, dt, nsub, rve.FP64, **law)
    eps_b, eps_n_b, R_b, p_b, y0_b = (t.cpu().numpy() for t in (*out, st_b))
    base = dict(e6=e6, en6=en6, ep6=ep6, v=v, al=al, R=R)
    grads = dict(e6=eps_b, en6=eps_n_b, ep6=y0_b[:6], v=y0_b[6:22].T, al=y0_b[22:].T, R=R_b.T.reshape(n, 3, 3))
    scales = dict(e6=1e-3, en6=1e-3, ep6=3e-4, v=1e-3, al=1e-3, R=1e-2)
    J = lambda m=mat, **ch: _J(m, *({**base, **ch}[k] for k in ("R", "en6", "e6", "ep6", "v", "al")), sb, yb, dt,  # noqa: E731
                               nsub)
    for name, x in base.items():
        d = np.random.default_rng(sum(map(ord, name))).normal(size=x.shape) * scales[name]
        num = (J(**{name: x + 1e-5 * d}) - J(**{name: x - 1e-5 * d})) / 2e-5
        ana = float(np.sum(grads[name] * d))
        assert abs(num - ana) <= 2e-6 * max(abs(num), abs(ana)) + 1e-10, (name, num, ana)
    for k, name in enumerate(PARAMS):
        p0 = getattr(mat, name)
        h = 1e-6 * max(abs(p0), 1.0)
        num = (J(dataclasses.replace(mat, **{name: p0 + h})) - J(dataclasses.replace(mat, **{name: p0 - h}))) / (2 * h)
        ana = float(np.sum(p_b[k]))
        assert abs(num - ana) <= 2e-5 * max(abs(num), abs(ana)) + 1e-8, (name, num, ana)
