"""The tune cache keeps batches with resident launches apart from batches of the
same sizes without them (GPU)."""
import numpy as np
import pytest

from paper_2508_09738_gb300 import binding as B
from paper_2508_09738_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_2508_09738_gb300 import build
    build.build()


def test_choice_without_resident_launches_is_not_taken_for_them(tmp_path):
    gs = [W.blobs_knn(n=700 + 50 * i, K=4, seed=i, label_frac=0.05) for i in range(5)]
    cache = str(tmp_path / "tune.txt")
    opts = {t: B.fw_seg_default_opts(max_iters=40, class_table=t) for t in ("off", "auto")}
    for t, resident in (("off", 0), ("auto", 5)):
        for tuned in (1, 2):
            with B.Batch(gs, opts[t], tune_cache=cache) as b:
                i = b.info()
                assert (i.tuned, i.resident) == (tuned, resident), t
                b.solve()
                if resident:
                    assert i.schedule == B.SCHED["items"]
                    for p, g in enumerate(gs):
                        with B.Segmenter(g, max_iters=40) as s:
                            s.solve()
                            assert np.array_equal(b.U(p), s.U())
