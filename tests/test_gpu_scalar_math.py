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
