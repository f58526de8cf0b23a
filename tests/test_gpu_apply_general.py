"""H*v of models whose interaction window spans several 8-site chunks (the
row kernel with the general diagonal): against the oracle on every row and
against the generic kernels, at the edges of its windows of 128 strings, with
two, three and four chunks, spin-flip / pair-hop moves beside several chunks, and
long hop lists.  Tolerances as for every H*v: 1e-12 norm-wise (FP64, DF64), one
rounding to float (FP32 vectors with double-float sums).
"""
import numpy as np
import pytest

import workloads as W
from oracle import sector as osec
from tests._gpu import empty_vec, ensure_built, rel_err, to_dev, to_host, torch_cuda

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def env():
    torch = torch_cuda()
    ed = ensure_built()
    ctx = ed.ed_ctx_create(0)
    yield ed, ctx, torch
    ed.ed_ctx_destroy(ctx)


def wide_kanamori(n_s, seed):
    """Kanamori impurity with a density interaction on the first bath site too,
    so that the interaction window covers every site."""
    m = W.kanamori(n_s, seed=seed)
    m.U_site[0] = 1.25
    return m


def dense_hops(n_s, seed):
    r = np.random.default_rng(seed)
    m = W.hubbard_cluster(n_s)
    # a few distinct matrix elements on every bond, exactly symmetric
    vals = r.choice([-1.0, -0.75, -0.5, 0.25], size=(n_s, n_s))
    m.T = np.triu(vals, 1) + np.triu(vals, 1).T + np.diag(r.uniform(-1, 1, n_s))
    return m


CASES = [("ring 11, 462 strings: generic", lambda: W.hubbard_cluster(11, tp=0.2), 2, 5, 0),
         ("ring 12, 792 strings", lambda: W.hubbard_cluster(12, tp=0.2), 3, 5, 1),
         ("ring 13, 1287 strings", lambda: W.hubbard_cluster(13), 1, 5, 1),
         ("ring 18, three chunks", lambda: W.hubbard_cluster(18, tp=0.1), 1, 3, 1),
         ("ring 26, four chunks", lambda: W.hubbard_cluster(26, tp=0.1), 1, 3, 1),
         ("impurity moves beside two chunks", lambda: wide_kanamori(12, 3), 4, 5, 1),
         ("every bond", lambda: dense_hops(12, 5), 2, 5, 1)]


@pytest.mark.parametrize("prec", ["fp64", "df64", "fp32"])
@pytest.mark.parametrize("name,mk,nu,nd,kern", CASES, ids=[c[0] for c in CASES])
def test_general_diagonal_row_kernel(env, name, mk, nu, nd, kern, prec):
    ed, ctx, torch = env
    m = mk()
    H = osec.build_csr(m, nu, nd)
    n = H.shape[0]
    x = W.random_vector(n, seed=9)
    xin = x.astype(np.float32).astype(np.float64) if prec == "fp32" else x
    ref = H @ xin
    xd = to_dev(x, prec, ed, torch)
    got = {}
    for flags in (0, ed.ED_SECTOR_GENERIC):
        sec = ed.ed_sector_create(ctx, m, nu, nd, prec, flags)
        try:
            if flags == 0:
                assert ed.ed_sector_get_info(sec).kernel == kern
                assert ed.ed_sector_autotune(sec, reps=1).n_candidates == 0   # nothing to tune
            yd = torch.full_like(empty_vec(n, prec, ed, torch), float("nan"))
            ed.ed_apply_h(sec, xd, yd)
            torch.cuda.synchronize()
            got[flags] = to_host(yd, prec, n, ed, torch)
        finally:
            ed.ed_sector_destroy(sec)
    tol = 2.0 ** -24 if prec == "fp32" else 1e-12
    assert rel_err(got[0], ref) <= tol
    assert rel_err(got[0], got[ed.ED_SECTOR_GENERIC]) <= tol


def test_general_row_kernel_in_the_solvers(env):
    """The row kernel's own <x, Hx> partials (general diagonal) through the
    reorthogonalised and the three-vector solver."""
    ed, ctx, torch = env
    m = W.hubbard_cluster(12, tp=0.15)
    H = osec.build_csr(m, 2, 5)
    import scipy.sparse.linalg as sla
    ref = float(sla.eigsh(H, k=1, which="SA", tol=1e-13)[0][0])
    for reorth in (True, False):
        sec = ed.ed_sector_create(ctx, m, 2, 5, "df64")
        try:
            ev, _, _ = ed.ed_lanczos(sec, k=1, tol=1e-10, max_iter=300, reorth=reorth)
            assert abs(ev[0] - ref) <= 1e-10 * abs(ref)
        finally:
            ed.ed_sector_destroy(sec)
