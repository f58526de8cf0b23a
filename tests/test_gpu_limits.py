"""What creating a sector costs, in time and in device memory."""
import time

import pytest

import workloads as W
from tests._gpu import ensure_built, torch_cuda

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def env():
    return ensure_built(), torch_cuda()


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
