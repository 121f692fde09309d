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


@pytest.mark.parametrize("ipl", [7, 16])
@pytest.mark.parametrize("weights,K,opts", [
    ("f64", 6, dict(tol_mode="rel", gap_tol=0.075, max_iters=400)),
    ("f64", 3, dict(step_rule="armijo", max_iters=60)),
    ("f64", 11, dict(max_iters=50, laplacian="comb")),
    ("f32", 2, dict(max_iters=50)), ("f32", 4, dict(max_iters=50, oracle="full")),
    ("bf16", 5, dict(max_iters=50, eps=0.3)), ("f32", 7, dict(max_iters=50, laplacian="comb")),
    ("f32", 8, dict(step_rule="armijo", max_iters=60)), ("f32", 9, dict(max_iters=50)),
    ("bf16", 16, dict(tol_mode="rel", gap_tol=0.1, max_iters=300))])
def test_fused_pass_a_equals_stepwise(weights, K, opts, ipl):
    """Captured graphs of fused iterations (the extra committing block, the
    quick step decision, two accumulator banks) against the same passes with
    k_finish between them: the same bits for every class count's pass A."""
    g = W.blobs_knn(n=3001, K=K, seed=20 + K, label_frac=0.03)
    kw = dict(weight_dtype=weights, class_table="off", **opts)
    with B.Segmenter(g, iters_per_launch=ipl, **kw) as a, B.Segmenter(g, **kw) as b:
        assert a.forms().solve == B.SOLVE["passes"]
        sa, sb = a.solve(), b.step(opts["max_iters"] + 1)
        assert same_stats(sa, sb)
        assert np.array_equal(a.U(), b.U())


@pytest.mark.parametrize("graph", ["required", "off"])
@pytest.mark.parametrize("weights", ["f32", "bf16", "f64"])
def test_item_launches_beside_resident_ones(weights, graph):
    """Problems of more than 16 classes run as per-item launches beside the
    resident launches of the others, in one captured graph or directly, in one
    launch or several, each with its own cap: every problem equals its own
    solve."""
    gs = [W.blobs_knn(n=1200, K=20, seed=1, label_frac=0.05), W.blobs_knn(n=2000, K=5, seed=2),
          W.sbm(n=17 * 900, K=17, deg_in=14.0, deg_out=3.0, seed=3), W.blobs_knn(n=257, K=3, seed=4),
          W.voronoi_image(side=61, K=5, seed=5, label_frac=0.02)]
    caps = [40, 25, 33, 0, 60]
    opts = [B.fw_seg_default_opts(max_iters=c, weight_dtype=weights) for c in caps]
    want = [alone(g, weight_dtype=weights, max_iters=c) for g, c in zip(gs, caps)]
    for per in (0, 7):
        with B.Batch(gs, opts, weight_dtype=weights, schedule="items", lanes_per_row=0,
                     blocks_per_sm=1, iters_per_launch=per, use_graph=graph) as b:
            assert b.info().resident == 3
            for _ in range(2):
                b.reset()
                stats = b.solve()
                for p in range(len(gs)):
                    assert np.array_equal(b.U(p), want[p][0]), p
                    assert np.array_equal(b.labels(p), want[p][1]), p
                    assert same_stats(stats[p], want[p][2]), p


@pytest.mark.parametrize("weights", ["f32", "bf16", "f64"])
def test_item_launches_of_every_class_bound(weights):
    """Per-item launches alone, one problem of each class bound, with stops at
    different iterations over several launches."""
    gs = [W.blobs_knn(n=500 + 211 * K, K=K, seed=40 + K, label_frac=0.05)
          for K in (2, 4, 5, 8, 9, 12, 13, 16, 24, 32)]
    o = [dict(max_iters=20 + 9 * p, tol_mode="rel", gap_tol=0.2 if p % 3 == 0 else 0.0,
              class_table="off") for p in range(len(gs))]
    with B.Batch(gs, [B.fw_seg_default_opts(weight_dtype=weights, **x) for x in o],
                 weight_dtype=weights, schedule="items", lanes_per_row=0, blocks_per_sm=1,
                 iters_per_launch=16) as b:
        assert b.info().resident == 0
        stats = b.solve()
        for p, g in enumerate(gs):
            U, lab, st = alone(g, weight_dtype=weights, **o[p])
            assert np.array_equal(b.U(p), U), p
            assert same_stats(stats[p], st), p


def test_served_lone_request_with_long_row_takes_the_class_table():
    """A row past the resident kernel's 1,020 entries, scattered columns and
    more tiles than SMs: the server's lone epochs run the class-table pass B,
    and equal the request's own solve."""
    base = W.sbm(n=50_000, K=5, deg_in=16.0, deg_out=3.0, label_frac=0.01, seed=81)
    rows = np.repeat(np.arange(base.n), np.diff(base.row_ptr))
    up = rows < base.col
    hub = np.arange(30, base.n, 37)                      # 1,351 neighbours of node 7
    i, j = np.concatenate([rows[up], np.full(hub.size, 7)]), np.concatenate([base.col[up], hub])
    rp, col, w = W.from_edges(base.n, i, j, np.ones(i.size))
    g = W.Graph(base.n, rp, col, w, base.K, base.labels, base.truth)
    o = dict(max_iters=150, gap_tol=1e-4, tol_mode="rel")
    with B.Segmenter(g, **o) as s:
        f = s.forms()
        assert f.class_table == 1 and f.solve == B.SOLVE["passes"]
    U, lab, st = alone(g, **o)
    with B.Server(hbm_budget_bytes=1 << 30, max_slots=4, max_K=8, iters_per_epoch=8) as srv:
        t = srv.submit(g, **o)
        rc, lab_s, st_s = srv.wait(t, g.n, timeout_ms=60_000)
        assert rc == st.status and np.array_equal(lab_s, lab) and same_stats(st_s, st)


def test_tuner_counts_iterations_not_the_start_of_resident_launches():
    """Twelve small problems that the resident kernel takes beside one that it
    does not: per-item and resident launches are a quarter faster over a solve,
    though not over its first iterations.  The tuner picks them."""
    gs = [W.blobs_knn(n=300, K=3, seed=9)] * 12 + [W.blobs_knn(n=300, K=20, seed=51)]
    for _ in range(3):
        with B.Batch(gs, B.fw_seg_default_opts(max_iters=200)) as b:
            i = b.info()
            assert (i.schedule, i.resident) == (B.SCHED["items"], 12)
