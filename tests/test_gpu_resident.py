"""The resident kernel (a whole solve in one launch) against the two-kernel
path driven step by step: the same iterates, labels and statistics bit for bit
(GPU).  Both take every sum in the same order and the quick step decision is
used only where it is provably the rounding of the FP64 one, so any difference
here is a bug, not rounding."""
import numpy as np
import pytest

from paper_2508_09738_gb300 import binding as B
from paper_2508_09738_gb300 import workloads as W

pytestmark = pytest.mark.gpu

STATS = ("iters", "status", "active_rows", "gap", "gap0", "q", "alpha", "objective")


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_2508_09738_gb300 import build
    build.build()


def check(g, resident=True, **opts):
    with B.Segmenter(g, **opts) as a, B.Segmenter(g, **opts) as b:
        sa = a.solve()
        sb = b.step(opts["max_iters"] + 1)
        assert (sa.launches == 1) == resident
        for f in STATS:
            assert getattr(sa, f) == getattr(sb, f), f
        assert np.array_equal(a.U(), b.U())
        assert np.array_equal(a.labels(), b.labels())
        # a second solve from the start, and a stepped one after a launch
        a.reset()
        assert a.solve().gap == sa.gap
        return sa


# one block, tile and layer edges, clusters, the cluster / grid line, ragged ends
@pytest.mark.parametrize("n,K,weights", [
    (40, 2, "f32"), (255, 3, "bf16"), (256, 3, "f32"), (257, 4, "f32"), (513, 5, "f32"),
    (1025, 6, "bf16"), (4097, 8, "f32"), (8193, 10, "f32"), (16384, 3, "f32"),
    (16385, 3, "bf16"), (30001, 9, "f32"), (2001, 11, "f32"), (2001, 13, "bf16"),
    (2001, 16, "f32"), (1237, 3, "f64"), (3000, 7, "f64"), (1300, 12, "f64")])
def test_sizes_and_classes(n, K, weights):
    g = W.sbm(n=n // K * K, K=K, deg_in=11.0, deg_out=3.0, label_frac=0.03, seed=n + K)
    check(g, weight_dtype=weights, max_iters=70)


@pytest.mark.parametrize("lanes", [1, 2, 4, 32])
@pytest.mark.parametrize("n", [3000, 40_000])
def test_lanes(lanes, n):
    g = W.sbm(n=n, K=5, deg_in=22.0, deg_out=3.0, label_frac=0.02, seed=lanes)
    check(g, weight_dtype="f32", max_iters=40, lanes_per_row=lanes)


@pytest.mark.parametrize("side,height,K", [(37, 41, 3), (300, 211, 4), (558, 557, 6)])
def test_images_walked_in_place(side, height, K):
    g = W.voronoi_image(side=side, height=height, K=K, label_frac=0.01, seed=side)
    check(g, weight_dtype="f32", max_iters=40, omega0=1e5)


@pytest.mark.parametrize("opts", [
    dict(laplacian="comb"), dict(step_rule="armijo"), dict(oracle="full"),
    dict(laplacian="comb", step_rule="armijo", oracle="full"), dict(eps=float("inf")),
    dict(eps=0.3), dict(tol_mode="rel", gap_tol=0.2), dict(gap_tol=1e-3), dict(omega0=0.0)])
def test_options(opts):
    g = W.blobs_knn(n=2500, K=6, seed=11, label_frac=0.03)
    check(g, weight_dtype="f32", max_iters=90, **opts)


def test_many_iterations_and_wide_columns():
    """Past the statistics ring (32 iterations) and on a graph of more than
    65,536 scattered rows (4-bit classes, 32-bit columns)."""
    check(W.blobs_knn(n=900, K=4, seed=3), weight_dtype="f32", max_iters=333)
    check(W.sbm(n=90_000, K=10, deg_in=16.0, deg_out=3.0, seed=9), weight_dtype="bf16",
          max_iters=50)


def test_where_it_does_not_apply():
    """K > 16, a row of more than 1,020 entries and an explicit pass B form
    keep the two-kernel path; its results do not change."""
    check(W.blobs_knn(n=1200, K=20, seed=4), resident=False, max_iters=30)
    n = 1500
    i = np.concatenate([np.zeros(n - 1, int), np.arange(1, n - 1)])
    j = np.concatenate([np.arange(1, n), np.arange(2, n)])
    rp, col, w = W.from_edges(n, i, j, np.ones(i.size))
    lab = np.full(n, -1, np.int32)
    lab[[3, n // 2]] = [0, 1]
    check(W.Graph(n, rp, col, w, 2, lab, lab), resident=False, max_iters=30)
    check(W.blobs_knn(n=1200, K=4, seed=4), resident=False, max_iters=30, class_table="off")


def test_solves_in_parts():
    """Warm start, refreshes and a raised position between solves: launches
    start from and leave the state of the two-kernel path."""
    g = W.blobs_knn(n=3001, K=5, seed=8, label_frac=0.03)
    rng = np.random.default_rng(1)
    U = rng.dirichlet(np.ones(5), size=g.n)
    with B.Segmenter(g, max_iters=60) as a, B.Segmenter(g, max_iters=60) as b:
        a.set_U(U)
        b.set_U(U)
        a.step(7)
        b.step(7)
        sa, sb = a.solve(), b.step(60)
        assert (sa.gap, sa.objective) == (sb.gap, sb.objective)
        assert np.array_equal(a.U(), b.U())
    with B.Segmenter(g, max_iters=64, refresh_every=16, iters_per_launch=16) as a, \
            B.Segmenter(g, max_iters=64, refresh_every=16, iters_per_launch=16,
                        class_table="off") as b:
        sa, sb = a.solve(), b.solve()
        assert (sa.iters, sa.gap, sa.objective) == (sb.iters, sb.gap, sb.objective)
        assert np.array_equal(a.U(), b.U())


# regular grids past the resident kernel: pass B and the one-shot pass from row
# patterns, against the column-reading forms (32-bit indices never use patterns)
@pytest.mark.parametrize("weights", ["f32", "bf16"])
@pytest.mark.parametrize("side,height,K,opts", [
    (601, 520, 4, {}), (601, 520, 2, dict(laplacian="comb")), (1031, 977, 3, {}),
    (640, 500, 8, dict(oracle="full")), (640, 500, 5, dict(eps=0.1)), (320, 1000, 7, {}),
    (2400, 2101, 6, {})])
def test_patterns_equal_columns(weights, side, height, K, opts):
    g = W.voronoi_image(side=side, height=height, K=K, label_frac=0.01, seed=side + K)
    kw = dict(weight_dtype=weights, max_iters=12, omega0=1e5, **opts)
    with B.Segmenter(g, **kw) as a, B.Segmenter(g, index_width=32, **kw) as b:
        assert a.forms().index_width == 16 and b.forms().index_width == 32
        assert np.array_equal(a.oneshot()[0], b.oneshot()[0])
        sa, sb = a.solve(), b.solve()
        for f in STATS:
            assert getattr(sa, f) == getattr(sb, f), f
        assert np.array_equal(a.U(), b.U())
        assert np.array_equal(a.labels(), b.labels())


def test_oneshot_on_a_resident_problem():
    g = W.voronoi_image(side=211, height=90, K=5, label_frac=0.02, seed=2)
    with B.Segmenter(g, eps=0.1, omega0=1e5) as a, \
            B.Segmenter(g, eps=0.1, omega0=1e5, index_width=32) as b:
        assert np.array_equal(a.oneshot()[0], b.oneshot()[0])
        assert a.solve().gap == b.solve().gap


@pytest.mark.parametrize("weights", ["f32", "f64"])
@pytest.mark.parametrize("n,K", [(33, 3), (16383, 4), (16384, 4), (16385, 4), (9362, 7), (9363, 7)])
def test_read_out_around_the_host_line(n, K, weights):
    """An iterate read back is the one written, exactly, on both sides of the
    line between the read-out on the host (fewer than 65,536 values) and the
    one on the device."""
    i = np.arange(n)
    rows = np.stack([(i - 1) % n, (i + 1) % n], 1)
    rows.sort(axis=1)
    g = W.Graph(n=n, row_ptr=np.arange(0, 2 * n + 1, 2, dtype=np.int32),
                col=rows.ravel().astype(np.int32), w=np.ones(2 * n), K=K,
                labels=np.where(i < K, i, -1).astype(np.int32), truth=(i % K).astype(np.int32))
    rng = np.random.default_rng(5)
    U = rng.integers(1, 64, (n, K)).astype(np.float64)
    U[:, 0] += 4096 - U.sum(1)
    U /= 4096.0     # multiples of 2^-12: exact in either type, rows sum to 1
    with B.Segmenter(g, weight_dtype=weights) as s:
        s.set_U(U)
        assert np.array_equal(s.U(), U)
