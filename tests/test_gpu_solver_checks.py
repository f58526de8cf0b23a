"""Convergence checks of the solvers: what a check reads, and what it costs."""
import numpy as np
import pytest
import scipy.sparse.linalg as sla

import workloads as W
from oracle import sector as osec
from tests._gpu import ensure_built, torch_cuda

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def env():
    torch = torch_cuda()
    ed = ensure_built()
    ctx = ed.ed_ctx_create(0)
    yield ed, ctx, torch
    ed.ed_ctx_destroy(ctx)


def test_rotations_of_the_projected_matrix_have_no_bias(env):
    """Values after some 200 rotations of each row of the projected matrix, whose
    roundings fall to both sides: sqrt(200) u on average, u = 2^-53, times three
    (200 u would be a drift)."""
    ed, ctx, torch = env
    err = []
    for seed in range(8):
        m = W.kanamori(8, seed=seed)
        H = osec.build_csr(m, 4, 4)
        X = sla.eigsh(H, k=4, which="SA", tol=1e-13)[1].astype(np.longdouble)   # Rayleigh quotients in extended precision
        ref = np.sort((X * (H.astype(np.longdouble) @ X)).sum(0) / (X * X).sum(0)).astype(np.float64)
        sec = ed.ed_sector_create(ctx, m, 4, 4, "fp64")
        ev, _, _ = ed.ed_lanczos_tr(sec, k=4, tol=1e-10, max_basis=40, max_iter=3000, check_every=5, seed=seed + 1)
        ed.ed_sector_destroy(sec)
        err.append(np.linalg.norm(ev - ref) / np.linalg.norm(ref))
    assert np.mean(err) <= 3 * 200 ** 0.5 * 2.0 ** -53, err
