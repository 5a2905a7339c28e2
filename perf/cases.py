"""Performance cases: what users of the solver have it do, through its public Python entry points.

Five kinds of work, each over the range of sizes, precisions and options that this
repository's workloads, tests and benchmark use:

  step      load increments of one RVE (RVE.step), then the fields of the new state
  ensemble  one load increment of several realizations at once (step_batch)
  points    the per-voxel constitutive update on its own (material_point), or its reverse
            pass (material_point_vjp)
  gradient  misfit and gradient of a load history (history_gradient)
  label     Voronoi labelling of a voxel grid (label_voronoi)

A solver's increments follow one another, as in a load history: every pass continues from
the state that the last one left.  `prepare` takes the RVE into the plastic regime first, and
single RVEs run a set number of fixed-point iterations per increment (the number that the
increment takes to the usual tolerance, or less to keep a pass short), so that passes at
different strains do the same work.
"""
import math

import numpy as np
import torch

from paper_2402_09996_gb300 import inputs, rve

# the paper's parameter set with the hardening terms of the paper workload (bench.py)
PAPER = dict(C33=183000.0, r0_ord=130.0, r0_sup=200.0, r0_twin=130.0, K=104.0, Kt=104.0, n=6.42, nt=6.42,
             Q_s=9.57, Q_b=10.5, Kc=1.45, fm=0.8, eta=1.0e4, c=0.0, d=0.0)
DEFAULT = dict(C11=183000.0, C12=74000.0, C13=74000.0, C33=178000.0, C44=105000.0, C66=78000.0,
               r0_ord=90.0, r0_sup=200.0, r0_twin=110.0, K=10.0, n=10.0, Kt=10.0, nt=10.0,
               Q_s=20.0, Q_b=20.0, b_s=5.0, b_b=5.0, h_diag=1.0, h_off=1.2, c=1.0e4, d=500.0,
               Kc=1.45, fm=0.8, eta=1.0e4)
PARAMS = ["r0_ord", "r0_sup", "r0_twin", "Q_s", "Q_b", "b_s", "b_b", "c", "d"]
FIELDS = (rve.FIELD_STRESS, rve.FIELD_STRAIN, rve.FIELD_EPS_P, rve.FIELD_V, rve.FIELD_ALPHA)


def _step(name, nz, ny, nx, grains, p_twin, precision, dt, steps, iters, pre, pre_dt, material="default",
          green="willot"):
    return {"name": name, "kind": "step", "nz": nz, "ny": ny, "nx": nx, "grains": grains, "p_twin": p_twin,
            "precision": precision, "material": material, "green": green, "dt": dt, "steps": steps, "iters": iters,
            "pre": pre, "pre_dt": pre_dt}


def listed():
    return [
        # the smallest workload (16^3, 8 untwinned grains, FP64, increments of 0.1 % strain):
        # a verification run, where latency counts
        _step("rve_16_fp64", 16, 16, 16, 8, 0.0, "fp64", 1.0, 1, 24, 4, 1.0),
        # the smallest ensemble size under the paper's increments (5e-6 strain each): few
        # iterations per increment, so launches, waits and the commit count
        _step("rve_64_fp32_small_increments", 64, 64, 64, 50, 0.5, "fp32", 0.005, 10, 8, 8, 0.5),
        # the ordinary single RVE (200 half-twinned grains, 0.05 % strain per increment)
        _step("rve_128_fp32", 128, 128, 128, 200, 0.5, "fp32", 0.5, 1, 56, 6, 0.5),
        # the paper's grid, material and increments (shortening; real exponent 6.42)
        _step("rve_256_fp32_paper", 256, 256, 256, 1920, 0.5, "fp32", 0.005, 2, 8, 8, 0.5, material="paper"),
        # the default precision on a grid without power-of-two lines
        _step("rve_48_fp64", 48, 48, 48, 20, 0.5, "fp64", 0.5, 1, 24, 6, 0.5),
        # odd line lengths (3^2 5, 3 5^2, 2^2 5^2), continuous-frequency Green operator
        _step("rve_ragged_fp32_ms", 45, 75, 100, 60, 0.5, "fp32", 0.5, 1, 16, 5, 0.5, green="ms"),
        # realizations of four sizes stepped together to the tolerance (Sec. 5 statistics)
        {"name": "ensemble_fp32", "kind": "ensemble", "sizes": "64,96,128,160", "grains": "50,125,241,400",
         "p_twin": 0.5, "dt": 0.5, "pre": 4},
        # the constitutive update on a list of points (material drivers, parameter studies)
        {"name": "points_fp32", "kind": "points", "n": 1000003, "precision": "fp32", "material": "default",
         "dt": 0.5, "reverse": False},
        {"name": "points_fp64", "kind": "points", "n": 20011, "precision": "fp64", "material": "default",
         "dt": 0.5, "reverse": False},
        # its reverse pass (gradients of point-wise objectives, tangents)
        {"name": "points_reverse_fp32", "kind": "points", "n": 100003, "precision": "fp32", "material": "default",
         "dt": 0.5, "reverse": True},
        # calibration: misfit and gradient of a short history
        {"name": "gradient_20_fp64", "kind": "gradient", "n": 20, "grains": 10, "p_twin": 0.5, "precision": "fp64",
         "increments": 3, "dt": 0.5, "iters": 24},
        # the grain map of the ordinary RVE, left on the GPU
        {"name": "label_128", "kind": "label", "nz": 128, "ny": 128, "nx": 128, "grains": 200, "p_twin": 0.5},
    ]


def draw(rng):
    def log_int(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    def line(lo, hi, even=False):
        n = log_int(lo, hi)
        while True:
            m = n
            for p in (2, 3, 5):
                while m % p == 0:
                    m //= p
            if m == 1 and not (even and n % 2):
                return n
            n += 1

    kind = rng.choice(["step", "step", "step", "ensemble", "points", "points", "gradient", "label"])
    p_twin = rng.choice([0.0, 0.5, 1.0])
    if kind == "step":
        precision = rng.choice(["fp32", "fp32", "fp64"])
        hi = 160 if precision == "fp32" else 48
        shape = [line(12, hi), line(12, hi), line(12, hi, even=True)]
        dt = rng.choice([0.005, 0.1, 0.5])
        steps, iters = (4, 8) if dt < 0.01 else (1, rng.randint(12, 32))
        return dict(_step("", *shape, max(2, shape[0] * shape[1] * shape[2] // rng.randint(4000, 10000)), p_twin,
                          precision, dt, steps, iters, 5, 0.5, material=rng.choice(["default", "paper"]),
                          green=rng.choice(["willot", "willot", "ms"])), name="")
    if kind == "ensemble":
        sizes = [line(24, 128, even=True) for _ in range(rng.randint(2, 5))]
        return {"name": "", "kind": kind, "sizes": ",".join(map(str, sizes)),
                "grains": ",".join(str(max(2, s ** 3 // 8000)) for s in sizes), "p_twin": p_twin, "dt": 0.5, "pre": 4}
    if kind == "points":
        precision, reverse = rng.choice(["fp32", "fp64"]), rng.random() < 0.4
        return {"name": "", "kind": kind, "n": log_int(100, 100000 if reverse or precision == "fp64" else 1000000),
                "precision": precision, "material": rng.choice(["default", "paper"]),
                "dt": rng.choice([0.005, 0.5, 1.0]), "reverse": reverse}
    if kind == "gradient":
        return {"name": "", "kind": kind, "n": line(8, 20, even=True), "grains": rng.randint(2, 12),
                "p_twin": p_twin, "precision": "fp64", "increments": rng.randint(2, 3), "dt": 0.5, "iters": 24}
    return {"name": "", "kind": "label", "nz": log_int(10, 200), "ny": log_int(10, 200), "nx": log_int(10, 200),
            "grains": log_int(1, 2000), "p_twin": p_twin}


# ------------------------------------------------------------------------------------
# inputs and passes
# ------------------------------------------------------------------------------------
def _dtype(case):
    return torch.float64 if case["precision"] == "fp64" else torch.float32


def _n_sub(dt):
    """Substeps of an increment: the smallest power of two with dt / n_sub <= 1/8 s."""
    n = 1
    while dt / n > 0.125 * (1.0 + 1e-12):
        n *= 2
    return n


def _load(case):
    """Uniaxial load along z: tension, or the paper's shortening."""
    return (0.0, 0.0, -1e-3 if case.get("material") == "paper" else 1e-3, 0.0, 0.0, 0.0)


def _labels(inp):
    return rve.label_voronoi(inp, out=torch.empty(inp.shape, dtype=torch.int32, device="cuda"))


def _grid_inputs(case, seed):
    return inputs.make_inputs((case["nz"], case["ny"], case["nx"]), case["grains"], case["p_twin"], seed)


def _point_inputs(case, seed, device="cuda"):
    """Random orientations, strains and states: a third of the points stay elastic."""
    n, t = case["n"], _dtype(case)
    g = torch.Generator(device=device).manual_seed(seed)

    def uniform(lo, hi, *shape):
        return lo + (hi - lo) * torch.rand(shape, generator=g, dtype=torch.float64, device=device)

    def normal(scale, *shape):
        return scale * torch.randn(shape, generator=g, dtype=torch.float64, device=device)

    scale = 3.0 if case["material"] == "paper" else 1.0
    euler = torch.stack([uniform(0, 2 * math.pi, n), torch.arccos(uniform(-1, 1, n)), uniform(0, 2 * math.pi, n)])
    R = _rotations(euler.T)
    shear = torch.tensor([1.0, 1.0, 1.0] + [math.sqrt(0.5)] * 3, dtype=torch.float64, device=device)[:, None]
    eps_n = normal(1.5e-3 * scale, 6, n) * shear
    eps = eps_n + normal(1.0e-3 * scale, 6, n) * shear * min(1.0, case["dt"] / 0.5)
    quiet = torch.where(uniform(0, 1, n) < 0.33, 0.1, 1.0)
    ep = normal(3e-4, 6, n) * shear
    ep[:3] -= ep[:3].mean(0)
    v = uniform(0, 2e-3, 16, n)
    v[12:] *= 0.1
    al = uniform(-1e-3, 1e-3, 12, n)
    out = {"R": R.reshape(n, 9), "eps_n": eps_n * quiet, "eps": eps * quiet, "state": torch.cat([ep, v, al])}
    if case["reverse"]:
        out["sigma_b"] = normal(1e-2, 6, n)
        out["state_b"] = normal(10.0, 34, n)
    return {k: x.to(t).contiguous() for k, x in out.items()}


def _gradient_inputs(case, seed):
    n = case["n"]
    inp = inputs.make_inputs((n, n, n), case["grains"], case["p_twin"], seed)
    target = 1.1 * 135e3 * 1e-3 * case["dt"] * np.minimum(np.arange(1, case["increments"] + 1), 2.5)
    return inp, target


def prepare(case, seed):
    kind = case["kind"]
    if kind == "step":
        inp = _grid_inputs(case, seed)
        solver = rve.RVE(_labels(inp), inp.euler, precision=rve.FP64 if case["precision"] == "fp64" else rve.FP32,
                         green=rve.GREEN_MS if case["green"] == "ms" else rve.GREEN_WILLOT,
                         fixed_iters=case["iters"])
        if case["material"] == "paper":
            solver.set_material(**PAPER)
        solver.set_mixed_load(Edot=_load(case), dt=case["pre_dt"])
        solver.step(case["pre"])
        if case["dt"] != case["pre_dt"]:
            solver.set_mixed_load(Edot=_load(case), dt=case["dt"])
            solver.step(2)
        out = [torch.empty((rve.FIELD_COMPONENTS[f],) + solver.shape, dtype=_dtype(case), device="cuda")
               for f in FIELDS]
        return {"case": case, "solver": solver, "out": out}
    if kind == "ensemble":
        solvers = []
        for k, (n, g) in enumerate(zip(case["sizes"].split(","), case["grains"].split(","))):
            inp = inputs.make_inputs((int(n),) * 3, int(g), case["p_twin"], seed * 16 + k)
            solver = rve.RVE(_labels(inp), inp.euler, precision=rve.FP32)
            solver.set_mixed_load(Edot=_load(case), dt=case["dt"])
            solvers.append(solver)
        rve.step_batch(solvers, case["pre"])
        out = [torch.empty((6,) + s.shape, dtype=torch.float32, device="cuda") for s in solvers]
        return {"case": case, "solvers": solvers, "out": out}
    if kind == "points":
        return {"case": case, "n_sub": _n_sub(case["dt"]), "in": _point_inputs(case, seed),
                "precision": rve.FP64 if case["precision"] == "fp64" else rve.FP32,
                "material": PAPER if case["material"] == "paper" else {}}
    if kind == "gradient":
        inp, target = _gradient_inputs(case, seed)
        return {"case": case, "grain_id": _labels(inp), "euler": inp.euler, "target": target}
    inp = _grid_inputs(case, seed)
    return {"case": case, "inputs": inp, "out": torch.empty(inp.shape, dtype=torch.int32, device="cuda")}


def _mean(record, key, case):
    return np.asarray(record[key], dtype=np.float64 if case.get("precision") == "fp64" else np.float32)


def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "step":
        solver = state["solver"]
        solver.step(case["steps"])
        rec = solver.effective()
        return {"fields": [solver.field(f, out=o) for f, o in zip(FIELDS, state["out"])],
                "S": _mean(rec, "S", case), "E": _mean(rec, "E", case)}
    if kind == "ensemble":
        rve.step_batch(state["solvers"], 1)
        return {"stress": [s.field(rve.FIELD_STRESS, out=o) for s, o in zip(state["solvers"], state["out"])],
                "S": [_mean(s.effective(), "S", case) for s in state["solvers"]]}
    if kind == "points":
        p = state["in"]
        if case["reverse"]:
            state_b = p["state_b"].clone()  # overwritten with the adjoint at t_n
            eps_b, eps_n_b, R_b, param_b = rve.material_point_vjp(
                p["R"], p["eps_n"], p["eps"], p["state"], p["sigma_b"], state_b, case["dt"], state["n_sub"],
                state["precision"], **state["material"])
            return [eps_b, eps_n_b, R_b, param_b, state_b]
        new = p["state"].clone()  # a trial update: the state at t_n is kept
        sigma = rve.material_point(p["R"], p["eps_n"], p["eps"], new, case["dt"], state["n_sub"], state["precision"],
                                   **state["material"])
        return [sigma, new]
    if kind == "gradient":
        J, g_params, g_euler, _ = rve.history_gradient(state["grain_id"], state["euler"], case["increments"],
                                                       case["dt"], state["target"], precision=rve.FP64,
                                                       Edot=_load(case), fixed_iters=case["iters"])
        return {"J": np.array([J]), "params": g_params, "euler": g_euler}
    return rve.label_voronoi(state["inputs"], out=state["out"])


# ------------------------------------------------------------------------------------
# work: per voxel and fixed-point iteration the state (46 values and the grain id) and one
# round trip of the six half spectra; 1100 flops per right-hand side with its 16 rate solves
# ------------------------------------------------------------------------------------
RHS = 1100


def _iteration_work(voxels, iterations, n_sub, size):
    return (voxels * iterations * (46 * size + 4 + 12 * size), voxels * iterations * (4 * n_sub * RHS + 200))


def work(case):
    kind = case["kind"]
    size = 8 if case.get("precision") == "fp64" else 4
    if kind == "step":
        nvox = case["nz"] * case["ny"] * case["nx"]
        b, f = _iteration_work(nvox, case["steps"] * case["iters"], _n_sub(case["dt"]), size)
        return {"bytes": b + 46 * size * nvox, "flops": f}
    if kind == "ensemble":
        nvox = sum(int(s) ** 3 for s in case["sizes"].split(","))
        b, f = _iteration_work(nvox, 56, _n_sub(case["dt"]), 4)  # about 56 iterations to the tolerance
        return {"bytes": b + 6 * 4 * nvox, "flops": f}
    if kind == "points":
        rhs = 4 * _n_sub(case["dt"])
        values = (9 + 6 + 6 + 34 + 6 + 34) + (6 + 6 + 9 + 9 + 34 if case["reverse"] else 40)
        return {"bytes": case["n"] * values * size, "flops": case["n"] * rhs * RHS * (3 if case["reverse"] else 1)}
    if kind == "gradient":
        nvox = case["n"] ** 3
        b, f = _iteration_work(nvox, case["increments"] * case["iters"], _n_sub(case["dt"]), size)
        # adjoint iterations: the linear law's 42 values; the reverse sweeps: seven seeds and the constraint
        adj = case["increments"] * (case["iters"] * nvox * (42 + 12) * size + 260 * size * nvox)
        return {"bytes": b + adj, "flops": f + case["increments"] * nvox * 4 * _n_sub(case["dt"]) * RHS * 9}
    nvox = case["nz"] * case["ny"] * case["nx"]
    return {"bytes": 4 * nvox + 24 * case["grains"], "flops": 8 * nvox}


# ------------------------------------------------------------------------------------
# 64-bit reference: the law (Sec. 3 and 4) and the fixed point in plain torch
# ------------------------------------------------------------------------------------
_N = [(1, 1, -1)] * 3 + [(-1, 1, 1)] * 3 + [(1, -1, 1)] * 3 + [(1, 1, 1)] * 3 + [(1, 1, -1), (-1, 1, 1), (1, -1, 1),
                                                                                 (1, 1, 1)]
_L = [(0, 1, 1), (1, 0, 1), (1, -1, 0), (0, -1, 1), (-1, 0, -1), (-1, -1, 0), (0, 1, 1), (1, 0, -1), (1, 1, 0),
      (0, 1, -1), (1, 0, -1), (1, -1, 0), (1, 1, 2), (-1, 1, -2), (1, -1, -2), (1, 1, -2)]
_IJ = [(0, 0), (1, 1), (2, 2), (1, 2), (0, 2), (0, 1)]


def _rotations(euler):
    """Bunge angles (n, 3) -> crystal-to-sample rotations (n, 3, 3)."""
    (c1, c, c2), (s1, s, s2) = euler.cos().unbind(-1), euler.sin().unbind(-1)
    return torch.stack([c1 * c2 - s1 * c * s2, -c1 * s2 - s1 * c * c2, s1 * s,
                        s1 * c2 + c1 * c * s2, -s1 * s2 + c1 * c * c2, -c1 * s,
                        s * s2, s * c2, c], dim=-1).reshape(-1, 3, 3)


def _schmid(device):
    """(16, 6) tensor components of sym(n x l) / (|n| |l|)."""
    n, l = np.array(_N, float), np.array(_L, float)
    n /= np.linalg.norm(n, axis=1, keepdims=True)
    l /= np.linalg.norm(l, axis=1, keepdims=True)
    m = 0.5 * (n[:, :, None] * l[:, None, :] + l[:, :, None] * n[:, None, :])
    return torch.tensor(np.stack([m[:, i, j] for i, j in _IJ], axis=1), device=device)


def _stiffness(m, device):
    C = torch.zeros((6, 6), dtype=torch.float64)
    C[0, 0] = C[1, 1] = m["C11"]
    C[2, 2] = m["C33"]
    C[0, 1] = C[1, 0] = m["C12"]
    C[0, 2] = C[2, 0] = C[1, 2] = C[2, 1] = m["C13"]
    C[3, 3] = C[4, 4] = 2 * m["C44"]
    C[5, 5] = 2 * m["C66"]
    return C.to(device)


def _tensor(v):
    return torch.stack([v[0], v[5], v[4], v[5], v[1], v[3], v[4], v[3], v[2]], dim=-1).reshape(-1, 3, 3)


def _six(t):
    return torch.stack([t[:, i, j] for i, j in _IJ])


def _power(z, n):
    if n != round(n):
        return z ** n
    out, b, k = None, z, int(n)
    while k:
        if k & 1:
            out = b if out is None else out * b
        b, k = b * b, k >> 1
    return torch.ones_like(z) if out is None else out


def _rate(a, P, K, n, eta):
    """rho = P <(a - eta rho) / K>^n: Newton from above in z = (a - eta rho) / K, the last step
    differentiable in a and P."""
    with torch.no_grad():
        on = (a > 0) & (P > 0)
        aa, PP = torch.where(on, a, 1.0), torch.where(on, P, 1.0)
        z = torch.minimum(aa / K, (aa / (eta * PP)) ** (1.0 / n))
        for _ in range(8):
            zn1 = _power(z, n - 1)
            z = z - ((eta * PP * zn1 + K) * z - aa) / (n * eta * PP * zn1 + K)
    grad = a.requires_grad or P.requires_grad
    aa, PP = (torch.where(on, a, 1.0), torch.where(on, P, 1.0)) if grad else (aa, PP)
    zn1 = _power(z, n - 1)
    z = z - ((eta * PP * zn1 + K) * z - aa) / (n * eta * PP.detach() * zn1 + K)
    return torch.where(on, PP * _power(z, n), 0.0)


class _Law:
    """The constitutive update on (components, n) tensors; parameters may be tensors (n,)."""

    def __init__(self, m, device):
        self.m, self.S, self.C = m, _schmid(device), _stiffness(m, device)
        self.W = torch.tensor([1.0, 1, 1, 2, 2, 2], dtype=torch.float64, device=device)
        self.kind = ["r0_ord" if s % 3 == 2 else "r0_sup" for s in range(12)]

    def rates(self, e, ep, v, al):
        m = self.m
        tau = (self.S * self.W) @ (self.C @ (e - ep))
        hs, ht = 1.0 - torch.exp(-m["b_s"] * v[:12]), 1.0 - torch.exp(-m["b_b"] * v[12:])
        dq = m["h_diag"] - m["h_off"]
        r0 = torch.stack([m[k] + 0.0 * v[0] for k in self.kind])
        rs = r0 + m["Q_s"] * (m["h_off"] * hs.sum(0) + dq * hs)
        rt = m["r0_twin"] + m["Q_b"] * (m["h_off"] * ht.sum(0) + dq * ht)
        f = math.sqrt(2.0) * v[12:].sum(0)
        te = tau[:12] - m["c"] * al
        one = torch.ones((), dtype=torch.float64, device=e.device)
        rho_s = _rate(te.abs() - rs, one, m["K"], m["n"], m["eta"])
        P = ((m["Kc"] / math.sqrt(2.0)) * torch.clamp(m["fm"] - f, min=0.0)).expand(4, -1)
        rho_t = _rate(tau[12:] - rt, P, m["Kt"], m["nt"], m["eta"])
        g = torch.where(te < 0, -rho_s, rho_s)
        dep = (1.0 - f) * (self.S[:12].T @ g) + self.S[12:].T @ rho_t
        return dep, torch.cat([rho_s, rho_t]), g - m["d"] * rho_s * al

    def update(self, R, eps_n, eps, y, dt, n_sub):
        """Sample-frame strains -> (sample-frame stress, (ep, v, al))."""
        e0, e1 = (_six(R.transpose(1, 2) @ _tensor(x) @ R) for x in (eps_n, eps))
        de, h = e1 - e0, dt / n_sub
        for k in range(n_sub):
            s = [k / n_sub, (k + 0.5) / n_sub, (k + 0.5) / n_sub, (k + 1.0) / n_sub]
            k1 = self.rates(e0 + s[0] * de, *y)
            k2 = self.rates(e0 + s[1] * de, *(a + 0.5 * h * b for a, b in zip(y, k1)))
            k3 = self.rates(e0 + s[2] * de, *(a + 0.5 * h * b for a, b in zip(y, k2)))
            k4 = self.rates(e0 + s[3] * de, *(a + h * b for a, b in zip(y, k3)))
            y = tuple(a + (h / 6.0) * (p + 2.0 * q + 2.0 * r + t) for a, p, q, r, t in zip(y, k1, k2, k3, k4))
        return _six(R @ _tensor(self.C @ (e1 - y[0])) @ R.transpose(1, 2)), y


class _Solver:
    """The Green-operator fixed point with a set number of iterations per increment."""

    def __init__(self, grain_id, euler, m, green, iters):
        self.device, self.shape, self.iters = grain_id.device, tuple(grain_id.shape), iters
        self.law = _Law(m, self.device)
        self.R = _rotations(torch.tensor(euler, device=self.device))[grain_id.reshape(-1).long()]
        n = grain_id.numel()
        zeros = lambda c: torch.zeros((c, n), dtype=torch.float64, device=self.device)  # noqa: E731
        self.eps, self.y, self.sigma = zeros(6), (zeros(6), zeros(16), zeros(12)), zeros(6)
        self.E, self.E_old, self.count = np.zeros(6), np.zeros(6), 0
        ev = np.linalg.eigvalsh(self.law.C.cpu().numpy())  # Mandel: the shear entries are 2 C44, 2 C66
        two_mu = 0.5 * (ev[0] + ev[-1])
        self.mu, self.lam = 0.5 * two_mu, two_mu / 3.0 - two_mu / 3.0
        self.kappa = self._kappa(green)

    def _kappa(self, green):
        nz, ny, nx = self.shape
        t = []
        for n, count in ((nx, nx // 2 + 1), (ny, ny), (nz, nz)):
            i = np.arange(count)
            if green == "willot":
                t.append((np.where(2 * i == n, 1.0, np.sin(np.pi * i / n)),
                          np.where(2 * i == n, 0.0, np.cos(np.pi * i / n))))
            else:
                f = np.where(2 * i == n, 0.0, np.where(i <= n // 2, i, i - n))
                t.append((2 * np.pi * f / n, np.ones(count)))
        (sx, cx), (sy, cy), (sz, cz) = [[torch.tensor(np.asarray(a, float), device=self.device) for a in p] for p in t]
        out = lambda a, b, c: a[:, None, None] * b[None, :, None] * c[None, None, :]  # noqa: E731
        return torch.stack([out(cz, cy, sx), out(cz, sy, cx), out(sz, cy, cx)])

    def _green(self, tau):
        """-Gamma0 : tau on the half spectrum (6, nz, ny, nx // 2 + 1)."""
        k = self.kappa
        k2 = (k * k).sum(0)
        k = k / torch.where(k2 > 0, k2, 1.0).sqrt()
        u = [k[0] * tau[0] + k[1] * tau[5] + k[2] * tau[4], k[0] * tau[5] + k[1] * tau[1] + k[2] * tau[3],
             k[0] * tau[4] + k[1] * tau[3] + k[2] * tau[2]]
        w = k[0] * u[0] + k[1] * u[1] + k[2] * u[2]
        coef = (self.lam + self.mu) / (self.mu * (self.lam + 2 * self.mu))
        g = torch.stack([(k[i] * u[j] + k[j] * u[i]) / (2 * self.mu) - coef * k[i] * k[j] * w for i, j in _IJ])
        return -g * (k2 > 0)

    def step(self, Edot, dt):
        """Component 33 strain-controlled, the other mean stresses zero."""
        wm = np.array([1.0, 1, 1] + [math.sqrt(2.0)] * 3)
        C0 = np.diag([2 * self.mu] * 6)
        C0[:3, :3] += self.lam
        free, n = [0, 1, 3, 4, 5], self.eps.shape[1]
        if self.count == 0:
            dm = np.array([0, 0, Edot[2] * dt, 0, 0, 0])
            dm[free] = -np.linalg.solve(C0[np.ix_(free, free)], C0[free, 2] * dm[2])
            dE = dm / wm
        else:
            dE = self.E - self.E_old
            dE[2] = Edot[2] * dt
        E = self.E + dE
        eps = self.eps + torch.tensor(dE, device=self.device)[:, None]
        for it in range(self.iters):
            sigma, y = self.law.update(self.R, self.eps, eps, self.y, dt, _n_sub(dt))
            if it + 1 == self.iters:
                break
            tau = sigma - 2 * self.mu * eps
            tau[:3] -= self.lam * eps[:3].sum(0)
            hat = self._green(torch.fft.rfftn(tau.reshape((6,) + self.shape), dim=(1, 2, 3)))
            Em = E * wm
            Em[free] -= np.linalg.solve(C0[np.ix_(free, free)], sigma.mean(1).cpu().numpy()[free] * wm[free])
            E = Em / wm
            hat[:, 0, 0, 0] = torch.tensor(E * n, device=self.device)
            eps = torch.fft.irfftn(hat, s=self.shape, dim=(1, 2, 3)).reshape(6, n)
        self.E_old, self.E, self.eps, self.y, self.sigma = self.E, E, eps, y, sigma
        self.count += 1


def _exact_points(case, seed, device="cuda"):
    p = {k: v.double() for k, v in _point_inputs(case, seed, device).items()}
    m = dict(DEFAULT, **(PAPER if case["material"] == "paper" else {}))
    y = (p["state"][:6], p["state"][6:22], p["state"][22:])
    if not case["reverse"]:
        sigma, y = _Law(m, device).update(p["R"].reshape(-1, 3, 3), p["eps_n"], p["eps"], y, case["dt"],
                                          _n_sub(case["dt"]))
        return [sigma, torch.cat(y)]
    out = []
    for i in range(0, case["n"], 50000):
        s = slice(i, min(i + 50000, case["n"]))
        R = p["R"][s].reshape(-1, 3, 3).clone().requires_grad_()
        eps_n, eps, state = (p[k][:, s].clone().requires_grad_() for k in ("eps_n", "eps", "state"))
        par = {k: torch.full((R.shape[0],), m[k], dtype=torch.float64, device=device, requires_grad=True)
               for k in PARAMS}
        sigma, y = _Law(dict(m, **par), device).update(R, eps_n, eps, (state[:6], state[6:22], state[22:]),
                                                       case["dt"], _n_sub(case["dt"]))
        J = (sigma * p["sigma_b"][:, s]).sum() + (torch.cat(y) * p["state_b"][:, s]).sum()
        g = torch.autograd.grad(J, [eps, eps_n, R, state] + [par[k] for k in PARAMS])
        out.append([g[0], g[1], g[2].reshape(-1, 9).T, torch.stack(g[4:]), g[3]])
    return [torch.cat(x, dim=1) for x in zip(*out)]


def exact(case, seed):
    if case["kind"] == "points":
        return _exact_points(case, seed)
    if case["kind"] != "step":
        return None
    increments = case["pre"] + case["steps"] + (2 if case["dt"] != case["pre_dt"] else 0)
    stages = case["iters"] * 4 * (case["pre"] * _n_sub(case["pre_dt"]) + (increments - case["pre"]) * _n_sub(case["dt"]))
    if case["nz"] * case["ny"] * case["nx"] * stages > 6e8:
        return None  # over about 20 seconds
    inp = _grid_inputs(case, seed)
    m = dict(DEFAULT, **(PAPER if case["material"] == "paper" else {}))
    solver = _Solver(_labels(inp), inp.euler, m, case["green"], case["iters"])
    for k in range(increments):
        solver.step(_load(case), case["pre_dt"] if k < case["pre"] else case["dt"])
    return {"fields": [x.reshape((-1,) + solver.shape) for x in (solver.sigma, solver.eps) + solver.y],
            "S": solver.sigma.mean(1).cpu().numpy(), "E": solver.E.copy()}
