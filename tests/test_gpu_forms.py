"""Which kernels a handle's solve and a batch's launches run, as the library
reports it (GPU)."""
import pytest

from paper_2508_09738_gb300 import binding as B
from paper_2508_09738_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_2508_09738_gb300 import build
    build.build()


def solve_form(g, **opts):
    with B.Segmenter(g, max_iters=3, **opts) as s:
        form = s.forms().solve
        assert (s.solve().launches == 1) == (form == B.SOLVE["resident"])
        return {v: k for k, v in B.SOLVE.items()}[form]


def test_forms_name_the_kernels_of_a_solve():
    knn = W.blobs_knn(n=1200, K=4, seed=4)
    assert solve_form(knn) == "resident"
    assert solve_form(knn, weight_dtype="f64") == "resident"
    assert solve_form(knn, class_table="off") == "passes"
    assert solve_form(W.blobs_knn(n=1200, K=20, seed=4)) == "passes"
    img = W.voronoi_image(side=601, height=520, K=4, label_frac=0.01, seed=1)
    assert solve_form(img) == "patterns" and solve_form(img, weight_dtype="bf16") == "patterns"
    assert solve_form(img, index_width=32) == "passes"
    assert solve_form(img, weight_dtype="f64") == "passes"
    assert solve_form(W.voronoi_image(side=601, height=520, K=9, seed=1)) == "passes"


def test_batch_counts_its_resident_problems():
    gs = [W.blobs_knn(n=700, K=K, seed=K) for K in (3, 20, 5, 8)]
    for schedule, want in (("items", 3), ("static", 0), ("dynamic", 0)):
        with B.Batch(gs, B.fw_seg_default_opts(max_iters=5), schedule=schedule, lanes_per_row=0,
                     blocks_per_sm=1, iters_per_launch=0) as b:
            b.solve()
            assert b.info().resident == want, schedule


def test_batch_info_counts_the_slices():
    """pool_bytes holds the resident kernel's copies of the graphs too: at
    least a column and a weight for every entry."""
    gs = [W.blobs_knn(n=4000, K=K, seed=K) for K in (3, 5, 8)]
    got = {}
    for table in ("auto", "off"):
        with B.Batch(gs, B.fw_seg_default_opts(max_iters=5, class_table=table), schedule="items",
                     lanes_per_row=0, blocks_per_sm=1, iters_per_launch=0) as b:
            got[table] = b.info().pool_bytes
    assert got["auto"] - got["off"] >= sum(g.nnz for g in gs) * (2 + 4)
