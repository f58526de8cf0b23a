"""Sector creation and solvers at the edge of a context's device budget, and what
creating a sector costs."""
import time

import numpy as np
import pytest

import workloads as W
from tests._gpu import empty_vec, ensure_built, rel_err, to_dev, to_host, torch_cuda

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def env():
    return ensure_built(), torch_cuda()


def least_budget(ed, call, hi):
    """Smallest budget (to 64 bytes) under which call(ctx) succeeds."""
    lo = 0
    while hi - lo > 64:
        mid = (lo + hi) // 2
        try:
            ctx = ed.ed_ctx_create(0, mid)
        except ed.EdError:
            lo = mid
            continue
        try:
            call(ctx)
            hi = mid
        except ed.EdError as e:
            assert "ED_ERR_OOM" in str(e), e
            lo = mid
        finally:
            ed.ed_ctx_destroy(ctx)
    return hi


def product(ed, torch, sec, x, prec, n):
    y = empty_vec(n, prec, ed, torch)
    ed.ed_apply_h(sec, to_dev(x, prec, ed, torch), y)
    torch.cuda.synchronize()
    return to_host(y, prec, n, ed, torch)


@pytest.mark.parametrize("prec", ["fp64", "df64", "fp32"])
def test_row_tables_never_refuse_a_general_sector(env, prec):
    """A cluster whose interaction spans several chunks needs no row-kernel tables:
    where they do not fit, the sector keeps the generic kernels."""
    ed, torch = env
    m = W.hubbard_cluster(12, tp=0.2)
    n = W.sector_dim(12, 6, 6)
    made = []

    def create(flags):
        def call(ctx):
            sec = ed.ed_sector_create(ctx, m, 6, 6, prec, flags)
            ed.ed_sector_destroy(sec)
        return call
    plain = least_budget(ed, create(ed.ED_SECTOR_GENERIC), 1 << 24)
    for budget in (plain, plain + 4096, plain + 40000, 1 << 24):
        ctx = ed.ed_ctx_create(0, budget)
        sec = ed.ed_sector_create(ctx, m, 6, 6, prec)
        made.append(product(ed, torch, sec, W.random_vector(n, seed=6), prec, n))
        ed.ed_sector_destroy(sec)
        ed.ed_ctx_destroy(ctx)
    tol = 2.0 ** -23 if prec == "fp32" else 1e-14
    assert max(rel_err(a, made[0]) for a in made) <= tol


@pytest.mark.parametrize("prec,tables", [("fp64", 629140), ("df64", 1229712), ("fp32", 1119120)])
def test_windows_cut_at_blocks_only_where_they_fit(env, prec, tables):
    """Windows that start anew at each impurity block take more tables than windows
    of 128 strings throughout (`tables` bytes for 13 sites); a budget for the
    latter is enough."""
    ed, torch = env
    m = W.kanamori(13, seed=1)
    n = W.sector_dim(13, 7, 6)
    ctx = ed.ed_ctx_create(0)
    base = ed.ed_ctx_bytes_in_use(ctx)
    x, made = W.random_vector(n, seed=6), []
    ed.ed_ctx_destroy(ctx)
    for budget in (base + tables, 1 << 24):
        ctx = ed.ed_ctx_create(0, budget)
        sec = ed.ed_sector_create(ctx, m, 7, 6, prec)
        made.append(product(ed, torch, sec, x, prec, n))
        assert ed.ed_sector_get_info(sec).kernel in (2, 4)
        ed.ed_sector_destroy(sec)
        ed.ed_ctx_destroy(ctx)
    assert rel_err(made[0], made[1]) <= (2.0 ** -23 if prec == "fp32" else 1e-14)


@pytest.mark.parametrize("prec", ["fp64", "df64", "fp32"])
@pytest.mark.parametrize("solver", ["full", "restart"])
def test_projections_need_no_room_beside_the_basis(env, solver, prec):
    """The reorthogonalised solvers run where the sector, the basis and the
    coefficients fit; without room for the projections' partial sums they go
    through the basis in smaller groups."""
    ed, torch = env
    m = W.kanamori(11, seed=3)
    dim, steps, k = W.sector_dim(11, 5, 6), 40, 2
    eb = 4 if prec == "fp32" else 8
    vec = (dim + 31) // 32 * 32 * eb
    out = {}

    def call(ctx):
        sec = ed.ed_sector_create(ctx, m, 5, 6, prec)
        call.held = ed.ed_ctx_bytes_in_use(ctx)
        try:
            if solver == "full":
                out["ev"] = ed.ed_lanczos(sec, k=k, tol=1e-300, max_iter=steps, check_every=steps, allow_not_converged=True)[0]
            else:
                out["ev"] = ed.ed_lanczos_tr(sec, k=k, tol=1e-300, max_basis=steps, keep=8, max_iter=steps,
                                             check_every=steps, allow_not_converged=True)[0]
        finally:
            ed.ed_sector_destroy(sec)
    least = least_budget(ed, call, 1 << 28)
    if solver == "full":     # 40 + 1 basis vectors, the work vector, up to 40 KB of coefficients
        room = (steps + 2) * vec + 40000
    else:                    # the same, 8 vectors to rotate into, four matrices of 128 rows
        room = (steps + 2 + 8) * vec + 4 * 128 * 128 * 8 + 40000
    assert least - call.held <= room, (least - call.held, room)
    ctx = ed.ed_ctx_create(0, least)
    call(ctx)
    ed.ed_ctx_destroy(ctx)
    tight = out["ev"]
    ctx = ed.ed_ctx_create(0)
    call(ctx)
    ed.ed_ctx_destroy(ctx)
    assert np.max(np.abs(tight - out["ev"])) <= (1e-5 if prec == "fp32" else 1e-11) * np.max(np.abs(out["ev"]))


def test_creating_a_general_sector_stays_cheap(env):
    """The row kernel's tables of a 15-site ring take no more than the sector's own
    (fastest of 30 creations each; 0.35 ms for the sector itself)."""
    ed, torch = env
    m = ed.Model(W.hubbard_cluster(15, tp=0.2))
    ctx = ed.ed_ctx_create(0)
    best = {}
    for flags in (0, ed.ED_SECTOR_GENERIC):
        for _ in range(30):
            t0 = time.perf_counter()
            sec = ed.ed_sector_create(ctx, m, 7, 8, "df64", flags)
            dt = time.perf_counter() - t0
            best[flags] = min(best.get(flags, dt), dt)
            ed.ed_sector_destroy(sec)
    ed.ed_ctx_destroy(ctx)
    assert best[0] <= 2.0 * best[ed.ED_SECTOR_GENERIC], best
