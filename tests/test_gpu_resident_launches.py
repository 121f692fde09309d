"""Launches of the resident kernel: their length, their bounded waits, and
what a caller learns when one runs out (GPU)."""
import time

import numpy as np
import pytest

from paper_2508_09738_gb300 import binding as B
from paper_2508_09738_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_2508_09738_gb300 import build
    build.build()


@pytest.mark.parametrize("per", [0, 1_000_000])
def test_batch_launches_hold_at_most_4096_iterations(per):
    """A batch ends its resident launches after 4,096 iterations as a handle
    does, and goes on with the next: the same bits as the handle's solve."""
    g = W.blobs_knn(n=300, K=3, seed=7, label_frac=0.05)
    o = dict(max_iters=9000, eps=float("inf"))     # convex: no early stop
    with B.Segmenter(g, **o) as s:
        st = s.solve()
        U = s.U()
    assert st.iters == 9000 and st.launches == 3
    with B.Batch([g], B.fw_seg_default_opts(**o), schedule="items", lanes_per_row=0,
                 iters_per_launch=per, blocks_per_sm=1) as b:
        sb = b.solve()[0]
        assert (sb.iters, sb.gap, sb.objective, sb.launches) == (9000, st.gap, st.objective, 3)
        assert np.array_equal(b.U(0), U)


# a cluster's exchange, a grid's barrier
@pytest.mark.parametrize("n", [3001, 30_001])
def test_wait_that_runs_out_in_a_handle(n):
    """Blocks that wait for more than ever arrives give up after 2 s: the
    solve reports it, nothing hangs, and a reset makes the handle usable."""
    g = W.blobs_knn(n=n, K=5, seed=3, label_frac=0.02)
    with B.Segmenter(g, max_iters=20, class_table="off") as s:
        want = s.step(20)
        U = s.U()
    with B.Segmenter(g, max_iters=20, test_barrier_extra=1) as s:
        t0 = time.time()
        with pytest.raises(B.FwError) as e:
            s.solve()
        assert e.value.status == B.FW_ERR_TIMEOUT
        assert 1.0 < time.time() - t0 < 10.0
        s.reset()
        st = s.step(20)          # the launches of the two passes have no such waits
        assert (st.gap, st.objective) == (want.gap, want.objective)
        assert np.array_equal(s.U(), U)


@pytest.mark.parametrize("n", [3001, 30_001])
def test_wait_that_runs_out_in_a_server(n):
    """spin_budget_ms bounds the waits of served resident launches; only the
    request concerned fails."""
    g = W.blobs_knn(n=n, K=5, seed=3, label_frac=0.02)
    with B.Segmenter(g, max_iters=20) as s:
        s.solve()
        lab = s.labels()
    with B.Server(hbm_budget_bytes=1 << 30, max_slots=4, max_K=8, spin_budget_ms=20) as srv:
        t0 = time.time()
        bad = srv.submit(g, max_iters=20, test_barrier_extra=1)
        good = srv.submit(g, max_iters=20)
        assert srv.wait(bad, g.n, timeout_ms=30_000)[0] == B.FW_ERR_TIMEOUT
        assert time.time() - t0 < 1.5
        rc, l, _ = srv.wait(good, g.n, timeout_ms=30_000)
        assert rc == B.FW_NOT_CONVERGED and np.array_equal(l, lab)
        assert srv.info().failed == 1


@pytest.mark.parametrize("graph", ["required", "off"])
@pytest.mark.parametrize("n", [3001, 30_001])
def test_wait_that_runs_out_in_a_batch(n, graph):
    """A batch does not report success for a problem whose launch gave up,
    whatever the others' statuses are, and says which kind of error it was."""
    g = W.blobs_knn(n=n, K=5, seed=3, label_frac=0.02)
    ok = W.blobs_knn(n=500, K=3, seed=4)
    opts = [B.fw_seg_default_opts(max_iters=20), B.fw_seg_default_opts(max_iters=20,
                                                                       test_barrier_extra=1),
            B.fw_seg_default_opts(max_iters=0)]
    with B.Batch([ok, g, ok], opts, schedule="items", lanes_per_row=0, blocks_per_sm=1,
                 iters_per_launch=0, spin_budget_ms=20, use_graph=graph) as b:
        t0 = time.time()
        with pytest.raises(B.FwError) as e:
            b.solve()
        assert time.time() - t0 < 1.5
        assert e.value.status == B.FW_ERR_TIMEOUT and "wait" in str(e.value)
        with B.Segmenter(ok, max_iters=20) as s:
            s.solve()
            assert np.array_equal(b.U(0), s.U())
    with B.Batch([ok, g], B.fw_seg_default_opts(max_iters=20), schedule="items", lanes_per_row=0,
                 blocks_per_sm=1, iters_per_launch=0, spin_budget_ms=20, test_barrier_extra=1) as b:
        with pytest.raises(B.FwError) as e:
            b.solve()
        assert e.value.status == B.FW_ERR_TIMEOUT


@pytest.mark.parametrize("opts", [{}, dict(refresh_every=8, iters_per_launch=8)])
def test_solve_goes_on_beside_kernels_that_keep_their_sms(opts):
    """A grid of resident blocks that cannot all be placed leaves without a
    trace, and the solve goes on beside the other kernels: it ends long before
    them, with the same bits as alone, and so does one under way when they end."""
    torch = pytest.importorskip("torch")
    g = W.voronoi_image(side=552, height=540, K=6, label_frac=0.01, seed=4)   # 1,165 tiles
    kw = dict(max_iters=200, omega0=1e5, **opts)
    others = [torch.cuda.Stream() for _ in range(16)]   # one block, one SM each
    with B.Segmenter(g, **kw) as s:
        alone = s.solve()
        U = s.U()
        for ms in (300, 3):
            s.reset()
            torch.cuda.synchronize()
            t0 = time.time()
            for o in others:
                with torch.cuda.stream(o):
                    torch.cuda._sleep(int(ms * 2e6))
            st = s.solve()
            if ms == 300:
                assert time.time() - t0 < 0.2
            assert (st.gap, st.objective, st.iters) == (alone.gap, alone.objective, alone.iters)
            assert np.array_equal(s.U(), U)
            torch.cuda.synchronize()
