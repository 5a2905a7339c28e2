"""Accuracy of single rates against the root of the regularised law in extended precision, over the
slip rates 2^-100 .. 2^20 per second (the tables of rate_table.cuh and the law constants beyond
them), and of the hardening exponential in double.

One point per rate, one substep, strain held, eps_23 the only strain: the eight slip systems
with a share of it are driven by exactly a = C e_23 (no resistance, no kinematic hardening), and
the time step is so short that the state moves by 2^-84 (float) or 2^-184 (double) at most, so
that all four stages see that a.  The kinematic variable (c = d = 0) then ends at
(h/6)(k + 2k + 2k + k): five roundings besides the rate's."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

LD = np.longdouble
EPS = {0: 2.0**-53, 1: 2.0**-24}  # unit roundoff by precision


def _root(a, K, n, eta):
    """rho of rho = ((a - eta rho)/K)^n, by Newton steps on eta z^n + K z = a from above."""
    a, K, n, eta = a.astype(LD), LD(K), LD(n), LD(eta)
    z = np.minimum(a / K, (a / eta) ** (1 / n))
    for _ in range(24):
        zn1 = z ** (n - 1)
        z = z - ((eta * zn1 + K) * z - a) / (n * eta * zn1 + K)
    return z**n


def _alpha_rate(cuda, prec, e23, v, dt, **law):
    """(alpha after the step) / dt of slip system 1, per point."""
    import torch

    from paper_2402_09996_gb300 import rve

    tdt = torch.float32 if prec else torch.float64
    m = len(e23)
    R = torch.eye(3, dtype=tdt, device=cuda).reshape(1, 9).repeat(m, 1)
    e = torch.zeros((6, m), dtype=tdt, device=cuda)
    e[3] = torch.tensor(e23, device=cuda)
    st = torch.zeros((34, m), dtype=tdt, device=cuda)
    st[6:18] = torch.tensor(v, device=cuda)
    rve.material_point(R, e, e, st, dt, 1, prec, **law)
    # system 1 ((1 1 -1)[1 0 1], the second) has a share of eps_23
    return np.abs(st[22 + 1].cpu().numpy().astype(LD)) / LD(dt)


SLIP_ONLY = dict(r0_twin=1e30, Q_s=0.0, Q_b=0.0, c=0.0, d=0.0)  # twins never flow


@pytest.mark.parametrize("prec,K,n,eta,tol", [
    # the tables: their stated bounds (float 2.1e-7, double 2.4e-16)
    *[(1, K, n, eta, 2.1e-7 + 5 * EPS[1]) for K in (1e-6, 10.0, 1e7) for n in (2.0, 2.5, 5.0, 10.0, 10.2)
      for eta in (1e-4, 1e4)],
    *[(0, K, n, eta, 2.4e-16 + 5 * EPS[0]) for K in (1e-6, 10.0, 1e12) for n in (2.0, 2.5, 5.0, 10.0, 10.2)
      for eta in (1e-4, 1e4)],
    # larger K in float: coefficients of the small rates would be subnormal, so the Newton solve;
    # the bound of the float path
    *[(1, K, 10.0, 1e4, 2e-4) for K in (1.1e7, 1e9, 1e12)],
])
def test_slip_rate_accuracy(lib, cuda, prec, K, n, eta, tol):
    T = np.float32 if prec else np.float64
    base = -100 if prec else -200
    c44 = K * 2.0**-10 * np.sqrt(6.0) / 2.0
    C = T(2.0 * c44 * (1.0 / np.sqrt(6.0)))  # the slip-scaled modulus as the host forms it
    rng = np.random.default_rng(3)
    # every table reaches 5 octaves above K's own
    a = 2.0 ** rng.uniform(np.log2(K) - 52.0, np.floor(np.log2(K)) + 5.0, 3000)
    e23 = (a / float(C)).astype(T)
    a = (C * e23).astype(T)
    rho = _root(a, K, n, eta)
    worst = 0.0
    for lo in range(-100, 20, 8):  # points whose alpha comes out near 2^base
        sel = (rho >= 2.0**lo) & (rho < 2.0 ** (lo + 8))
        if not sel.any():
            continue
        got = _alpha_rate(cuda, prec, e23[sel], np.zeros(int(sel.sum()), T), 2.0 ** (base - lo), K=K, n=n, eta=eta,
                          C44=c44, r0_ord=0.0, r0_sup=0.0, **SLIP_ONLY)
        worst = max(worst, float(np.max(np.abs(got / rho[sel] - 1))))
    assert worst <= tol, worst


def test_hardening_exponential_in_double(lib, cuda):
    """A resistance of -exp(-b v) (r0 + Q (1 - e) with r0 = -1, Q = 1, h_diag = 1, h_off = 0) drives a
    system by a = exp(-b v), beside a stress of 2^-110 that only fixes the direction of flow (at
    none the stages would flow to and fro).  The square law passes the exponential's relative
    error on at most twice; its argument is the exact product, which the kernel's fused operations see."""
    rng = np.random.default_rng(4)
    v = np.concatenate([rng.uniform(0.0, 24.0, 1000), np.arange(0, 1024) / 64.0 * np.log(2.0)])
    a = LD(2.0) ** (LD(-1.44269504088896340736) * v.astype(LD))
    K, n, eta = 1.0, 2.0, 1e-4
    F = _root(a, K, n, eta)
    law = {**SLIP_ONLY, "Q_s": 1.0}
    worst = 0.0
    for lo in range(-100, 4, 8):
        sel = (F >= 2.0**lo) & (F < 2.0 ** (lo + 8))
        if sel.any():
            got = _alpha_rate(cuda, 0, np.full(int(sel.sum()), 2.0**-127), v[sel], 2.0 ** (-200 - lo), K=K, n=n, eta=eta,
                              r0_ord=-1.0, r0_sup=-1.0, b_s=1.0, h_diag=1.0, h_off=0.0, **law)
            worst = max(worst, float(np.max(np.abs(got / F[sel] - 1))))
    # exponential: table entry and last operation half a unit each, remainder 2^-54; rate as above
    assert worst <= 2 * (2 * EPS[0] + 2.0**-54) + 2.4e-16 + 5 * EPS[0], worst
