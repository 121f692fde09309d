"""fw_energy_noalloc at every class count around the shared-memory limits of
its kernel, K ascending in a process of its own: no earlier call with more
classes can have raised the kernel's limit (GPU)."""
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

CHILD = """
import numpy as np, torch
import oracle as O
from paper_2508_09738_gb300 import binding as B, workloads as W
for K in (2, 3, 9, 10, 11, 12, 13, 16, 31, 32):
    g = W.blobs_knn(n=1100, K=K, seed=60 + K, label_frac=0.05)
    U = np.random.default_rng(K).dirichlet(np.ones(K), size=g.n)
    d = [torch.from_numpy(np.ascontiguousarray(a, dtype=t)).cuda()
         for a, t in ((g.row_ptr, np.int32), (g.col, np.int32), (g.w, np.float64),
                      (U, np.float64), (g.labels, np.int32))]
    for lap in ("sym", "comb"):
        E_o = O.energy(U, O.make_problem(g, 50.0, 1000.0, "f64", kind=lap))
        E = B.fw_energy_noalloc(g.n, K, d[0].data_ptr(), d[1].data_ptr(), d[2].data_ptr(), g.nnz,
                                d[3].data_ptr(), K, d[4].data_ptr(), 50.0, 1000.0, lap)
        assert abs(E - E_o) <= 1e-12 * abs(E_o), (K, lap, E, E_o)
print("ok")
"""


def test_energy_of_every_class_count_in_a_new_process():
    pytest.importorskip("torch")
    from paper_2508_09738_gb300 import build
    build.build()
    r = subprocess.run([sys.executable, "-c", CHILD], cwd=ROOT, capture_output=True, text=True,
                       timeout=300, env=dict(os.environ, PYTHONPATH=ROOT))
    assert r.returncode == 0 and r.stdout.strip().endswith("ok"), r.stdout + r.stderr
