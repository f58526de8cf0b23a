"""Full reorthogonalisation of the Lanczos solvers at the edges of its tiles.

The projection kernels work on tiles of 512 elements (1024 floats), 8 vectors
per warp and round of 64, and at most 2048 basis vectors per launch.  Sector
dimensions below, at and just past one and two tiles, and bases shorter and
longer than a round and than one launch, against the oracle's dense spectrum.

Eigenvalues of an orthogonal Krylov basis are those of H to the format's
rounding: n_terms * u * ||H|| with u = 2^-53, 2^-46 and 2^-24, ||H|| < 30 and a
factor of 100 for the few hundred steps, relative to the value.  Orthonormality
of the returned vectors is that of a twice-projected basis, 100 u.
"""
import numpy as np
import pytest

import workloads as W
from oracle import sector as osec
from tests._gpu import empty_vec, ensure_built, to_host, torch_cuda

pytestmark = pytest.mark.gpu

U = {"fp64": 2.0 ** -53, "df64": 2.0 ** -46, "fp32": 2.0 ** -24}
SECTORS = [(3, 1, 1), (8, 1, 3), (8, 1, 4), (9, 2, 7), (9, 1, 4), (8, 4, 3), (8, 4, 4)]   # 9 .. 4900 states


@pytest.fixture(scope="module")
def env():
    torch = torch_cuda()
    ed = ensure_built()
    ctx = ed.ed_ctx_create(0)
    yield ed, ctx, torch
    ed.ed_ctx_destroy(ctx)


@pytest.mark.parametrize("prec", ["fp64", "df64", "fp32"])
@pytest.mark.parametrize("solver", ["full", "restart"])
@pytest.mark.parametrize("n_s,nu,nd", SECTORS)
def test_reorthogonalised_solvers_at_tile_edges(env, n_s, nu, nd, solver, prec):
    ed, ctx, torch = env
    m = W.kanamori(n_s, seed=21, n_orb=min(3, n_s - 1)) if n_s > 3 else W.aim(n_s, seed=21)
    H = osec.build_csr(m, nu, nd)
    n = H.shape[0]
    ref = np.linalg.eigvalsh(H.toarray())
    k = min(4, n)
    tol = {"fp64": 1e-10, "df64": 1e-10, "fp32": 1e-5}[prec]
    sec = ed.ed_sector_create(ctx, m, nu, nd, prec)
    try:
        v = empty_vec(n, prec, ed, torch, count=k)
        if solver == "full":
            ev, _, _ = ed.ed_lanczos(sec, k=k, tol=tol, max_iter=min(n, 400), check_every=10, evecs=v)
        else:
            ev, _, _ = ed.ed_lanczos_tr(sec, k=k, tol=tol, max_basis=min(n, 40), max_iter=3000, evecs=v)
        scale = max(1.0, np.max(np.abs(ref)))
        bound = 100 * 30 * U[prec] * scale
        assert np.all(np.abs(ev - ref[:k]) <= bound), (ev, ref[:k])
        X = to_host(v, prec, n * k, ed, torch).reshape(k, n)
        assert np.max(np.abs(X @ X.T - np.eye(k))) <= 100 * max(U[prec], 2.0 ** -53 * n ** 0.5)
        # a Ritz pair's residual is what the tolerance allows plus the product's rounding
        R = H @ X.T - X.T * ev
        assert np.max(np.linalg.norm(R, axis=0)) <= 2 * tol * scale + bound
    finally:
        ed.ed_sector_destroy(sec)


def test_basis_longer_than_one_launch(env):
    """2,100 basis vectors of the 4,900-state sector: the projections run range
    by range, and the whole basis stays orthogonal (no ghost copies: the lowest
    30 values are the oracle's, each once)."""
    ed, ctx, torch = env
    m = W.kanamori(8, seed=22)
    H = osec.build_csr(m, 4, 4)
    ref = np.linalg.eigvalsh(H.toarray())
    sec = ed.ed_sector_create(ctx, m, 4, 4, "fp64")
    try:
        ev, info, _ = ed.ed_lanczos(sec, k=30, tol=1e-300, max_iter=2100, check_every=2100, allow_not_converged=True)
        assert info.iters == 2100
        assert np.all(np.abs(ev - ref[:30]) <= 1e-11 * np.max(np.abs(ref))), np.max(np.abs(ev - ref[:30]))
    finally:
        ed.ed_sector_destroy(sec)


@pytest.mark.parametrize("power", [-20, 0, 40])
def test_tridiagonal_solver_scales(env, power):
    """The tridiagonal eigensolver scales its matrix by a power of two: the
    spectrum of 2^p H is 2^p times that of H, for p of both signs (whole Krylov
    space, so nothing depends on the residual tolerance)."""
    ed, ctx, torch = env
    m = W.aim(6, seed=3)
    H = osec.build_csr(m, 3, 2)
    ref = np.linalg.eigvalsh(H.toarray())[:6] * 2.0 ** power
    m.T, m.U_site = m.T * 2.0 ** power, m.U_site * 2.0 ** power
    sec = ed.ed_sector_create(ctx, m, 3, 2, "fp64")
    try:
        ev, _, _ = ed.ed_lanczos(sec, k=6, tol=1e-300, max_iter=H.shape[0], check_every=H.shape[0],
                                 allow_not_converged=True)
        assert np.all(np.abs(ev - ref) <= 1e-12 * np.max(np.abs(ref))), ev - ref
    finally:
        ed.ed_sector_destroy(sec)


@pytest.mark.parametrize("m_b", [5, 6, 39, 40, 112, 113, 127, 128])
def test_projected_eigensolver_sizes(env, m_b):
    """Thick restart with every kind of projected matrix: odd (padded by a zero
    row) and even, the vectors in shared memory (up to 112 rows) or in global
    scratch.  Values to 1e-12 ||H|| (FP64 rounding over a few hundred rotations
    of entries below 30), vectors orthonormal to 1e-12, residuals as the
    tolerance allows."""
    ed, ctx, torch = env
    m = W.aim(8, seed=4)
    H = osec.build_csr(m, 4, 3)
    n, k, tol = H.shape[0], 3, 1e-10
    ref = np.linalg.eigvalsh(H.toarray())
    scale = np.max(np.abs(ref))
    sec = ed.ed_sector_create(ctx, m, 4, 3, "fp64")
    try:
        v = empty_vec(n, "fp64", ed, torch, count=k)
        ev, _, _ = ed.ed_lanczos_tr(sec, k=k, tol=tol, max_basis=m_b, max_iter=20000, check_every=5, evecs=v)
        assert np.all(np.abs(ev - ref[:k]) <= 1e-12 * scale), ev - ref[:k]
        X = v.cpu().numpy().reshape(k, n)
        assert np.max(np.abs(X @ X.T - np.eye(k))) <= 1e-12
        assert np.max(np.linalg.norm(H @ X.T - X.T * ev, axis=0)) <= 2 * tol * max(1.0, scale)
    finally:
        ed.ed_sector_destroy(sec)
