"""The two-pass kernels where the resident kernel would take the problem, and
beside it: class_table other than "auto" and K > 16 keep a problem on them
(GPU)."""
import numpy as np
import pytest

from paper_2508_09738_gb300 import binding as B
from paper_2508_09738_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_2508_09738_gb300 import build
    build.build()


def alone(g, **opts):
    with B.Segmenter(g, **opts) as s:
        st = s.solve()
        return s.U(), s.labels(), st


def same_stats(a, b):
    return (a.iters, a.status, a.gap, a.q, a.alpha, a.objective) == \
        (b.iters, b.status, b.gap, b.q, b.alpha, b.objective)


@pytest.mark.parametrize("table", ["off", "on"])
def test_batches_and_server_keep_class_table_problems_out_of_resident_launches(table):
    gs = [W.blobs_knn(n=900, K=3, seed=5), W.sbm(n=50_000, K=5, deg_in=16.0, deg_out=3.0, seed=6)]
    want = [alone(g, max_iters=40) for g in gs]
    for tables, resident in (((table, table), 0), (("auto", table), 1), (("auto", "auto"), 2)):
        opts = [B.fw_seg_default_opts(max_iters=40, class_table=t) for t in tables]
        with B.Batch(gs, opts, schedule="items", lanes_per_row=0, blocks_per_sm=1,
                     iters_per_launch=0) as b:
            stats = b.solve()
            assert b.info().resident == resident
            for p in range(2):
                assert np.array_equal(b.U(p), want[p][0])
                assert same_stats(stats[p], want[p][2])
    with B.Server(hbm_budget_bytes=1 << 30, max_slots=4, max_K=8, iters_per_epoch=8) as srv:
        for order in ((1,), (0, 1), (1, 0)):   # alone: with the table; together: shared epochs
            tk = [(p, srv.submit(gs[p], max_iters=40, class_table=table)) for p in order]
            for p, t in tk:
                rc, lab, st = srv.wait(t, gs[p].n, timeout_ms=60_000)
                assert np.array_equal(lab, want[p][1]) and same_stats(st, want[p][2])
