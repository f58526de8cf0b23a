"""Convergence checks of the solvers: what a check reads, and what it costs."""
import numpy as np
import pytest
import scipy.sparse.linalg as sla

import workloads as W
from oracle import greens as og
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


@pytest.mark.parametrize("n_s", [9, 10, 11, 12, 13])   # norm partials of 7 to 152 blocks
def test_check_and_next_step_form_the_same_beta(env, n_s):
    """beta_1 of the three-vector recurrence as a check after one step reads it (the
    residual of a 1 x 1 problem) and as the second step forms it (the continued
    fraction's coefficients, the same start vector): the same bits."""
    ed, ctx, torch = env
    m = W.aim(n_s, seed=2)
    nu, nd, depth = n_s // 2 - 1, n_s // 2, 3
    C, (tu, td) = og.op_matrix(n_s, nu, nd, m.orb0, 0, True)
    sec = ed.ed_sector_create(ctx, m, tu, td, "fp64")
    try:
        for seed in range(4):
            x = W.random_vector(C.shape[1], seed=seed)
            _, co = ed.ed_greens_cf(ctx, m, "fp64", [(nu, nd, -1.0, torch.from_numpy(x).cuda())], 40.0, 1,
                                    orbital=m.orb0, depth=depth, want_coeffs=True)
            _, info, _ = ed.ed_lanczos(sec, k=1, tol=1e-300, max_iter=1, check_every=1, reorth=False,
                                       v0=torch.from_numpy(C @ x).cuda(), allow_not_converged=True)
            assert info.residual[0] == co[0][2 + depth + 1], (seed, info.residual[0], co[0][2 + depth + 1])
    finally:
        ed.ed_sector_destroy(sec)


@pytest.mark.parametrize("name,mk,nu,nd", [("impurity", lambda: W.aim(8, seed=4), 4, 3),
                                           ("kanamori", lambda: W.kanamori(8, seed=4), 4, 3),
                                           ("ring", lambda: W.hubbard_cluster(8, U=4.0, tp=0.1), 4, 4)])
@pytest.mark.parametrize("offset", ["none", "shift", "strong U"])
def test_restarted_checks_see_convergence_in_time(env, name, mk, nu, nd, offset):
    """A thick restart whose basis never fills builds the Krylov space of the plain
    solver, so its checks find the k lowest pairs converged after the same number
    of products, rounded up to the check interval: also where the eigenvalues lie
    far from zero or far apart beside the gaps of the wanted ones."""
    ed, ctx, torch = env
    m = mk()
    if offset == "shift":       # 2^14 per electron
        m.T = m.T + 2.0 ** 14 * np.eye(m.n_s)
    elif offset == "strong U":
        m.U_site = m.U_site + 2.0 ** 12 * (m.U_site != 0)
    every = 4
    sec = ed.ed_sector_create(ctx, m, nu, nd, "fp64")
    try:
        for k in (1, 2, 4):
            for tol in (1e-10, 1e-13):
                _, full, _ = ed.ed_lanczos(sec, k=k, tol=tol, max_iter=124, check_every=every, seed=3,
                                           allow_not_converged=True)
                _, tr, _ = ed.ed_lanczos_tr(sec, k=k, tol=tol, max_basis=128, max_iter=124, check_every=every, seed=3,
                                            allow_not_converged=True)
                assert tr.restarts == 0 and tr.iters <= -(-full.iters // every) * every, (k, tol, full.iters, tr.iters)
    finally:
        ed.ed_sector_destroy(sec)


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


@pytest.mark.parametrize("prec", ["fp64", "df64"])
def test_batched_basis_longer_than_one_launch(env, prec):
    """2,100 steps of a batch: its projections run range by range (at most 2,048
    vectors a launch) while a smaller sector beside it has long been exhausted.
    Lowest values, each once, as the oracle's dense spectrum and the single-sector
    solver give them: 1e-11 ||H|| (a few thousand roundings of 2^-46 ||H||)."""
    ed, ctx, torch = env
    m = W.kanamori(8, seed=22)
    sectors = [(4, 4), (2, 1), (3, 3)]      # 4,900, 224 and 3,136 states
    k, steps = 16, 2100
    b = ed.ed_batch_create(ctx, m, sectors, prec)
    try:
        ev = ed.ed_batch_lanczos(b, len(sectors), k=k, tol=1e-300, max_iter=steps, check_every=steps,
                                 allow_not_converged=True)[0]
    finally:
        ed.ed_batch_destroy(b)
    for q, (nu, nd) in enumerate(sectors):
        ref = np.linalg.eigvalsh(osec.build_csr(m, nu, nd).toarray())
        assert np.all(np.abs(ev[q] - ref[:k]) <= 1e-11 * np.max(np.abs(ref))), (q, np.max(np.abs(ev[q] - ref[:k])))
    sec = ed.ed_sector_create(ctx, m, 4, 4, prec)
    try:
        one, _, _ = ed.ed_lanczos(sec, k=k, tol=1e-300, max_iter=steps, check_every=steps, allow_not_converged=True)
        assert np.all(np.abs(ev[0] - one) <= 1e-11 * np.max(np.abs(ref)))
    finally:
        ed.ed_sector_destroy(sec)


@pytest.mark.parametrize("solver", ["full", "restart", "batch"])
def test_float_projections_at_tile_edges(env, solver):
    """Float vectors: eigenvalues to 100 u ||H|| (u = 2^-24, a few hundred roundings
    that mostly cancel), so that an error of 1e-4 in the projections shows."""
    ed, ctx, torch = env
    m = W.kanamori(8, seed=21)
    u = 2.0 ** -24
    for nu, nd in ((1, 4), (4, 3), (4, 4)):        # 560 states (one tile and 48), 3,920, 4,900
        ref = np.linalg.eigvalsh(osec.build_csr(m, nu, nd).toarray())
        n, k = len(ref), 4
        if solver == "batch":
            b = ed.ed_batch_create(ctx, m, [(nu, nd)], "fp32")
            ev = ed.ed_batch_lanczos(b, 1, k=k, tol=1e-5, max_iter=400, check_every=10)[0][0]
            ed.ed_batch_destroy(b)
        else:
            sec = ed.ed_sector_create(ctx, m, nu, nd, "fp32")
            if solver == "full":
                ev, _, _ = ed.ed_lanczos(sec, k=k, tol=1e-5, max_iter=400, check_every=10)
            else:
                ev, _, _ = ed.ed_lanczos_tr(sec, k=k, tol=1e-5, max_basis=40, max_iter=3000)
            ed.ed_sector_destroy(sec)
        assert np.max(np.abs(ev - ref[:k])) <= 100 * u * np.max(np.abs(ref)), (ev, ref[:k])
