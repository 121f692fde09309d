"""FP64 problems give a block one 256-row tile, so a cluster can have blocks
without rows: 3 tiles on 4 blocks, 5 to 7 on 8, 9 to 15 on 16.  They take part
in the exchange of totals; the iterates and statistics are those of the two
passes bit for bit (GPU)."""
import numpy as np
import pytest

from paper_2508_09738_gb300 import binding as B
from paper_2508_09738_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_2508_09738_gb300 import build
    build.build()


# tiles: blocks without rows
@pytest.mark.parametrize("tiles", [3, 4, 5, 7, 9, 12, 15, 16])
def test_blocks_without_rows(tiles):
    g = W.blobs_knn(n=256 * tiles - 9, K=4, seed=tiles, label_frac=0.05)
    o = dict(weight_dtype="f64", max_iters=300)
    with B.Segmenter(g, class_table="off", **o) as s:
        want = s.step(301)
        U = s.U()
    with B.Segmenter(g, **o) as s:
        assert s.forms().solve == B.SOLVE["resident"]
        for _ in range(3):
            st = s.solve()
            assert st.launches == 1
            assert (st.iters, st.gap, st.objective, st.q) == (want.iters, want.gap,
                                                              want.objective, want.q)
            assert np.array_equal(s.U(), U)
            s.reset()


@pytest.mark.parametrize("n", [700, 1237])
def test_a_wait_that_runs_out_beside_blocks_without_rows(n):
    g = W.blobs_knn(n=n, K=3, seed=n, label_frac=0.05)
    with B.Segmenter(g, weight_dtype="f64", max_iters=20, test_barrier_extra=1) as s:
        with pytest.raises(B.FwError) as e:
            s.solve()
        assert e.value.status == B.FW_ERR_TIMEOUT
        s.reset()
        assert s.step(5).iters == 5
