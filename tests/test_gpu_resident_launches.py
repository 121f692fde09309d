"""Launches of the resident kernel: their length, their bounded waits, and
what a caller learns when one runs out (GPU)."""
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
