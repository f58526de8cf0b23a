"""The scalar FP64 arithmetic of the solvers' serial chains against exact values.

Every input is chosen so that the quantity is reached exactly up to the one
operation under test, and every bound counts the roundings of that operation
(u = 2^-53 relative each).
"""
from decimal import Decimal, getcontext
from fractions import Fraction as F

import numpy as np
import pytest

import workloads as W
from tests._gpu import ensure_built, torch_cuda

pytestmark = pytest.mark.gpu

getcontext().prec = 60


@pytest.fixture(scope="module")
def env():
    torch = torch_cuda()
    ed = ensure_built()
    ctx = ed.ed_ctx_create(0)
    yield ed, ctx, torch
    ed.ed_ctx_destroy(ctx)


@pytest.mark.parametrize("power", [-36, 0, 70])   # 70: the sum of squares leaves a float's range
@pytest.mark.parametrize("reorth", [True, False])
def test_first_beta_is_rounded_once(env, reorth, power):
    """One step from a basis state of a star of one electron: H v - alpha v is the
    row of hops, whose squares add up exactly, so beta_1 (the residual after one
    step) is the square root rounded once: u."""
    ed, ctx, torch = env
    r = np.random.default_rng(11)
    n, worst = 24, 0.0
    for _ in range(20):
        T = np.zeros((n, n))
        h = r.integers(1, 2000, n - 1) / 64.0 * 2.0 ** power
        T[0, 1:] = T[1:, 0] = h
        T[0, 0] = 0.5 * 2.0 ** power
        sec = ed.ed_sector_create(ctx, W.Model(n, T, np.zeros(n)), 1, 0, "fp64")
        try:
            v0 = torch.zeros(n, dtype=torch.float64, device="cuda")
            v0[0] = 1.0
            _, info, _ = ed.ed_lanczos(sec, k=1, tol=1e-300, max_iter=1, check_every=1, v0=v0, reorth=reorth,
                                       allow_not_converged=True)
        finally:
            ed.ed_sector_destroy(sec)
        v = sum(F(float(x)) ** 2 for x in h)
        root = (Decimal(v.numerator) / Decimal(v.denominator)).sqrt()
        worst = max(worst, float(abs(Decimal(info.residual[0]) / root - 1) * 2 ** 53))
    assert worst <= 1.0 + 1e-9, worst


@pytest.mark.parametrize("scale", [1.0, 1e-25, 1e25, 1e160])   # inside and outside the squares' float range
def test_one_level_fraction(env, scale):
    """G of one empty site of energy zero is 1 / z, one reciprocal c - i d over q =
    c^2 + d^2: u/2 of q from the smaller square, u from the sum, u from the
    quotient; and over many z no less accurate than Smith's division."""
    ed, ctx, torch = env
    r = np.random.default_rng(12)
    n = 4096
    z = (r.standard_normal(n) + 1j * np.abs(r.standard_normal(n)) * 10.0 ** r.uniform(-2, 2, n)) * scale
    psi = torch.ones(1, dtype=torch.float64, device="cuda")
    G = ed.ed_greens_cf_z(ctx, W.Model(1, np.zeros((1, 1)), np.zeros(1)), "fp64", [(0, 0, 0.0, psi)], z, 1.0, depth=1)
    c, d = z.real, z.imag
    big = np.abs(c) >= d
    with np.errstate(over="ignore"):
        t = np.where(big, d / c, c / d)
        den = np.where(big, c + d * t, c * t + d)
        smith = np.where(big, 1 / den, t / den) - 1j * np.where(big, t / den, 1 / den)
    err = {"G": [], "smith": []}
    for i in range(n):
        cf, df = F(float(c[i])), F(float(d[i]))
        q = cf * cf + df * df
        for name, g in (("G", G[i]), ("smith", smith[i])):
            err[name] += [float(abs(F(float(g.real)) * q / cf - 1) * 2 ** 53), float(abs(F(float(g.imag)) * q / -df - 1) * 2 ** 53)]
    rms = {k: float(np.sqrt(np.mean(np.square(v)))) for k, v in err.items()}
    if scale == 1.0:
        assert max(err["G"]) <= 2.5 + 1e-9, max(err["G"])
    assert rms["G"] <= 1.02 * rms["smith"], rms   # 2%: four times the spread of a mean over 8,192 roundings
