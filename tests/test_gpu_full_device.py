"""Calls on a device whose memory is all taken (GPU).  In processes of their
own, so that nothing else runs short."""
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

START = """
import numpy as np, torch
from paper_2508_09738_gb300 import binding as B, workloads as W

g = W.blobs_knn(n=22_470, K=7, seed=1)
b = B.Batch([g], B.fw_seg_default_opts(max_iters=20), lanes_per_row=0)
s = B.Segmenter(g, max_iters=20)
b.solve(), s.solve()
U, G, lab = b.U(0), s.grad()[0], b.labels(0)
keep = []
for size in (4 << 30, 256 << 20, 16 << 20, 2 << 20):
    try:
        while True:
            keep.append(torch.empty(size, dtype=torch.uint8, device="cuda"))
    except torch.OutOfMemoryError:
        pass
"""


def run(child):
    pytest.importorskip("torch")
    from paper_2508_09738_gb300 import build
    build.build()
    r = subprocess.run([sys.executable, "-c", START + child + 'print("ok")'], cwd=ROOT,
                       capture_output=True, text=True, timeout=600,
                       env=dict(os.environ, PYTHONPATH=ROOT))
    assert r.returncode == 0 and r.stdout.strip().endswith("ok"), r.stdout + r.stderr


def test_failed_create_leaves_no_error_to_the_next_call():
    """A create that fails (here already at its stream) is reported once, and
    not again by the launch checks of the calls that follow."""
    run("""
handles, failed = [], 0
gr = W.blobs_knn(n=300, K=16, seed=2)
try:
    while len(handles) < 2000:
        handles.append(B.Segmenter(gr))
except B.FwError:
    failed += 1
    assert np.array_equal(b.U(0), U)
    assert np.array_equal(s.grad()[0], G)
assert failed > 0
""")


def test_read_outs_need_no_device_memory():
    """With the library's own reserve used up as well, U and the gradient come
    back through the host."""
    run("""
def ring(n, K):
    i = np.arange(n)
    rows = np.stack([(i - 1) % n, (i + 1) % n], 1)
    rows.sort(axis=1)
    return W.Graph(n=n, row_ptr=np.arange(0, 2 * n + 1, 2, dtype=np.int32),
                   col=rows.ravel().astype(np.int32), w=np.ones(2 * n), K=K,
                   labels=np.where(i < K, i, -1).astype(np.int32), truth=(i % K).astype(np.int32))

handles = []
stream = torch.cuda.default_stream().cuda_stream or 2     # 2: the per-thread default stream
for n in (3_000_000, 300_000, 30_000, 3_000, 300):
    gr = ring(n, 16)
    try:
        while len(handles) < 2000:
            handles.append(B.Segmenter(gr, cuda_stream=stream))
    except B.FwError:
        pass
assert len(handles) < 2000
assert np.array_equal(b.U(0), U) and np.array_equal(b.labels(0), lab)
assert np.array_equal(s.grad()[0], G)
""")
