"""Performance cases of the segmentation library: what its users have it do.

A user builds a sparse similarity graph, labels a few nodes and asks for a
segmentation: one graph solved to the iteration cap on a handle that stays
(`Segmenter`), a new graph from host arrays to labels, the one-shot variant,
many small graphs in one batch, a burst of requests to the server, or the
objective of data that is already on the device.  Inputs are seeded synthetic
graphs of the three families of `paper_2508_09738_gb300/workloads.py` (k-NN
blobs, stochastic block models, 8-neighbour Voronoi images), generated on the
GPU so that fresh ones are cheap; sizes, class counts and solver options are
those of that module's CONFIGS, of the benchmark and of the tests, with odd
and ragged ones between them.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2508_09738_gb300 import binding as B
from paper_2508_09738_gb300 import workloads as W

DEV = "cuda"
L2_BYTES = 126 * 2**20      # what the card keeps on chip between two iterations


# ------------------------------------------------------------------- cases --

def listed():
    return [
        # A small network (the size of the paper's Amazon / LastFM graphs):
        # 2,000 points, 10-NN, 5 classes, 500 iterations.  Latency and launches.
        dict(name="knn2k_f32", kind="knn", n=2000, K=5, iters=500, weights="f32"),
        # The FP64 path, which the library offers for small problems and
        # checks, on a ragged size with few classes.
        dict(name="knn1k_f64", kind="knn", n=1237, K=3, iters=200, weights="f64"),
        # A mid-size network (Facebook-like, 2*10^4 nodes), more classes.
        dict(name="knn22k_f32", kind="knn", n=22470, K=7, iters=500, weights="f32"),
        # The large-network benchmark: block model, 200,000 nodes, 10 classes.
        dict(name="sbm200k_f32", kind="sbm", n=200_000, K=10, deg=22.0, iters=500,
             weights="f32"),
        # A photograph-sized image with odd sides, six classes.
        dict(name="image613x487_f32", kind="image", width=613, height=487, K=6, iters=200,
             weights="f32"),
        # A one-megapixel image with 16-bit weights, as the server gets them.
        dict(name="image1024_bf16", kind="image", width=1024, height=1024, K=4, iters=200,
             weights="bf16"),
        # The headline: the 2048 x 2048 image, 4 classes, 200 iterations.
        dict(name="image2048_f32", kind="image", width=2048, height=2048, K=4, iters=200,
             weights="f32"),
        # One-Shot Frank-Wolfe on the same image at the paper's image eps.
        dict(name="oneshot2048_f32", kind="oneshot", width=2048, height=2048, K=4,
             weights="f32"),
        # A new picture every call: graph on the host in, labels out, handle
        # created and destroyed (the path of a program that sees each graph once).
        dict(name="newgraph800x601_f32", kind="newgraph", width=800, height=601, K=5, iters=100,
             weights="f32"),
        # Many small graphs in one batch with 16-bit weights: the batched
        # benchmark's recipe (sizes log-uniform, 3 to 10 classes), 30 problems.
        dict(name="batch30_bf16", kind="batch", P=30, n_min=1000, n_max=60_000, iters=200,
             weights="bf16"),
        # A burst of requests to the server, blobs and images mixed, stopping
        # at g <= 1e-4 g_0 or after 500 iterations.
        dict(name="serve12_f32", kind="serve", P=12, n_min=1000, n_max=30_000, side_max=400,
             iters=500, weights="f32"),
        # The objective of device-resident data without an allocation.
        dict(name="energy300k_f64", kind="energy", n=300_007, K=6, deg=14.0),
    ]


def _logint(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """One more case of the listed ranges."""
    kind = rng.choice(["knn", "knn", "sbm", "image", "image", "oneshot", "newgraph", "batch",
                       "serve", "energy"])
    c = dict(kind=kind)
    if kind == "knn":
        n = _logint(rng, 300, 60_000)
        c.update(n=n, K=rng.choice([2, 3, 4, 5, 7, 8, 10, 11, 13, 16, 20]),
                 iters=rng.choice([100, 300, 500]),
                 weights=rng.choice(["f32", "f32", "bf16", "f64"] if n < 5000
                                    else ["f32", "f32", "bf16"]),
                 laplacian=rng.choice(["sym", "sym", "sym", "comb"]),
                 step_rule=rng.choice(["exact", "exact", "exact", "armijo"]),
                 oracle=rng.choice(["greedy", "greedy", "greedy", "full"]))
    elif kind == "sbm":
        c.update(n=_logint(rng, 10_000, 200_000), K=rng.choice([4, 5, 8, 10, 12]),
                 deg=rng.uniform(11.0, 22.0), iters=rng.choice([200, 500]),
                 weights=rng.choice(["f32", "bf16"]))
    elif kind in ("image", "oneshot", "newgraph"):
        top = 2048 if kind != "newgraph" else 1000
        wd = _logint(rng, 64, top)
        ht = min(top, max(48, int(wd * rng.uniform(0.6, 1.4))))
        c.update(width=wd, height=ht, K=rng.choice([3, 4, 4, 5, 6, 8] if wd * ht < 1 << 21
                                                   else [3, 4]),
                 weights=rng.choice(["f32", "bf16"]))
        if kind != "oneshot":
            c["iters"] = rng.choice([100, 200])
    elif kind == "batch":
        c.update(P=rng.randint(3, 30), n_min=400, n_max=_logint(rng, 4000, 60_000),
                 iters=rng.choice([60, 200]), weights=rng.choice(["f32", "bf16"]))
    elif kind == "serve":
        c.update(P=rng.randint(1, 12), n_min=500, n_max=30_000, side_max=rng.randint(100, 400),
                 iters=rng.choice([200, 500]), weights=rng.choice(["f32", "bf16"]))
    else:
        c.update(n=_logint(rng, 2000, 300_000), K=rng.randint(2, 8), deg=rng.uniform(6.0, 16.0),
                 laplacian=rng.choice(["sym", "comb"]))
    return c


# ------------------------------------------------------------------ inputs --

def _gen(seed):
    g = torch.Generator(device=DEV)
    g.manual_seed(int(seed) & 0x7FFFFFFF)
    return g


def _labels(truth, K, frac, gen):
    """A random fraction of the nodes keeps its class, at least one per class."""
    n = truth.numel()
    lab = torch.where(torch.rand(n, generator=gen, device=DEV) < frac, truth,
                      torch.full_like(truth, -1))
    first = torch.full((K,), n, dtype=torch.int64, device=DEV)
    first.scatter_reduce_(0, truth, torch.arange(n, device=DEV), "amin")
    first = first[first < n]
    lab[first] = truth[first]
    return lab


def _from_pairs(n, i, j, w):
    """Symmetric CSR of undirected pairs (duplicates merged, no self loops)."""
    keep = i != j
    lo, hi = torch.minimum(i, j)[keep], torch.maximum(i, j)[keep]
    key, inv = torch.unique(lo * n + hi, return_inverse=True)
    ww = torch.empty(key.numel(), dtype=torch.float64, device=DEV)
    ww[inv] = w[keep]          # duplicates carry equal weights
    lo, hi = key // n, key % n
    both, order = torch.sort(torch.cat([lo * n + hi, hi * n + lo]))
    ww = torch.cat([ww, ww])[order]
    rows = both // n
    rp = torch.zeros(n + 1, dtype=torch.int64, device=DEV)
    rp[1:] = torch.cumsum(torch.bincount(rows, minlength=n), 0)
    return rp.to(torch.int32), (both % n).to(torch.int32), ww


def _knn_dev(n, K, gen, knn=10, rank=7):
    """K Gaussian blobs in R^10, union-symmetrised 10-NN, self-tuning weights."""
    centres = 2.0 * torch.randn(K, 10, generator=gen, device=DEV, dtype=torch.float64)
    truth = (torch.arange(n, device=DEV) * K) // n
    X = centres[truth] + torch.randn(n, 10, generator=gen, device=DEV, dtype=torch.float64)
    Xf = X.float()
    sq = (Xf * Xf).sum(1)
    idx = torch.empty(n, knn, dtype=torch.int64, device=DEV)
    for a in range(0, n, 8192):
        b = min(n, a + 8192)
        d2 = sq[a:b, None] + sq[None, :] - 2.0 * (Xf[a:b] @ Xf.T)
        ar = torch.arange(b - a, device=DEV)
        d2[ar, ar + a] = float("inf")
        idx[a:b] = torch.topk(d2, knn, dim=1, largest=False).indices
    ii = torch.arange(n, device=DEV).repeat_interleave(knn)
    jj = idx.reshape(-1)
    lo, hi = torch.minimum(ii, jj), torch.maximum(ii, jj)
    d2 = ((X[lo] - X[hi]) ** 2).sum(1)
    own = ((X[:, None, :] - X[idx]) ** 2).sum(2).sort(1).values
    sig = own[:, rank - 1].sqrt().clamp_min(1e-12)
    w = torch.exp(-d2 / (sig[lo] * sig[hi]))
    return _from_pairs(n, ii, jj, w), truth


def _sbm_dev(n, K, deg, gen):
    """Block model: expected degree `deg`, ten in-block edges per cross edge."""
    m = n // K
    truth = torch.clamp(torch.arange(n, device=DEV) // m, max=K - 1)
    e_in, e_out = int(n * deg * 10 / 22), int(n * deg / 22)
    blk = torch.randint(0, K, (e_in,), generator=gen, device=DEV) * m
    i = blk + torch.randint(0, m, (e_in,), generator=gen, device=DEV)
    j = blk + torch.randint(0, m, (e_in,), generator=gen, device=DEV)
    i2 = torch.randint(0, n, (e_out,), generator=gen, device=DEV)
    j2 = torch.randint(0, n, (e_out,), generator=gen, device=DEV)
    i, j = torch.cat([i, i2]), torch.cat([j, j2])
    ok = i != j
    i, j = i[ok], j[ok]
    lone = (torch.bincount(i, minlength=n) + torch.bincount(j, minlength=n) == 0).nonzero()[:, 0]
    i, j = torch.cat([i, lone]), torch.cat([j, (lone + 1) % n])
    return _from_pairs(n, i, j, torch.ones(i.numel(), dtype=torch.float64, device=DEV)), truth


def _image_dev(width, height, K, gen):
    """Noisy piecewise-constant RGB image, 8-neighbour graph in raster order."""
    n = width * height
    f64 = dict(device=DEV, dtype=torch.float64)
    seeds = torch.rand(K, 2, generator=gen, **f64) * torch.tensor([height, width], **f64)
    colours = torch.rand(K, 3, generator=gen, **f64)
    yy = (torch.arange(height, **f64) + 0.5)[:, None, None]
    xx = (torch.arange(width, **f64) + 0.5)[None, :, None]
    truth = ((yy - seeds[:, 0]) ** 2 + (xx - seeds[:, 1]) ** 2).argmin(2).reshape(-1)
    img = colours[truth] + 0.1 * torch.randn(n, 3, generator=gen, **f64)
    ids = torch.arange(n, device=DEV).reshape(height, width)
    dst = torch.full((n, 8), -1, dtype=torch.int64, device=DEV)
    off = [(-1, -1), (-1, 0), (-1, 1), (0, -1), (0, 1), (1, -1), (1, 0), (1, 1)]
    d3 = dst.view(height, width, 8)
    for t, (dy, dx) in enumerate(off):
        y0, y1 = max(0, -dy), height - max(0, dy)
        x0, x1 = max(0, -dx), width - max(0, dx)
        d3[y0:y1, x0:x1, t] = ids[y0 + dy:y1 + dy, x0 + dx:x1 + dx]
    ok = dst >= 0
    rp = torch.zeros(n + 1, dtype=torch.int64, device=DEV)
    rp[1:] = torch.cumsum(ok.sum(1), 0)
    src = torch.arange(n, device=DEV).repeat_interleave(rp[1:] - rp[:-1])
    dst = dst[ok]
    s = torch.zeros(dst.numel(), **f64)
    for ch in range(3):
        d = img[src, ch] - img[dst, ch]
        s += d * d
    return (rp.to(torch.int32), dst.to(torch.int32), torch.exp(-s / 0.05)), truth


# label fractions and solver parameters of the three families (CONFIGS)
_FRAC = dict(knn=0.05, sbm=0.01, image=0.005)


def _dev_graph(family, case, seed):
    """((row_ptr, col, w), labels, K) on the device."""
    gen = _gen(seed)
    K = case["K"]
    if family == "knn":
        csr, truth = _knn_dev(case["n"], K, gen)
    elif family == "sbm":
        csr, truth = _sbm_dev(case["n"], K, case["deg"], gen)
    else:
        csr, truth = _image_dev(case["width"], case["height"], K, gen)
    return csr, _labels(truth, K, _FRAC[family], gen), K


def _host_graph(dev):
    (rp, col, w), lab, K = dev
    lab = lab.to(torch.int32).cpu().numpy()
    rp = rp.cpu().numpy()
    return W.Graph(rp.size - 1, rp, col.cpu().numpy(), w.cpu().numpy(), K, lab, lab)


def _members(case, seed):
    """The (family, case) list of a batch or a burst: sizes and class counts
    belong to the case (spread log-uniformly), the data to the seed."""
    out = []
    P = case["P"]
    for p in range(P):
        f = ((p * 0.6180339887) % 1.0) if P > 1 else 0.5
        n = int(case["n_min"] * (case["n_max"] / case["n_min"]) ** f)
        if case["kind"] == "serve" and p % 2:
            side = int(64 * (case["side_max"] / 64) ** f)
            out.append(("image", dict(width=side + 1, height=side, K=3 + p % 6)))
        else:
            out.append(("knn", dict(n=n, K=3 + (5 * p) % 8)))
    return [(fam, c, seed * 1000 + p) for p, (fam, c) in enumerate(out)]


def _opts(family, case):
    o = dict(eps=50.0, omega0=1e5 if family == "image" else 1000.0,
             weight_dtype=case["weights"])
    if case["kind"] == "oneshot":
        o["eps"] = 0.1
    else:
        o["max_iters"] = case["iters"]
    if case["kind"] == "serve":
        o.update(tol_mode="rel", gap_tol=1e-4)
    for k in ("laplacian", "step_rule", "oracle"):
        if k in case:
            o[k] = case[k]
    return o


_FAMILY = dict(knn="knn", sbm="sbm", image="image", oneshot="image", newgraph="image",
               energy="sbm")


class _Server(B.Server):
    def __del__(self):
        try:
            self.close()
        except Exception:
            pass


def prepare(case, seed):
    kind = case["kind"]
    if kind == "batch":
        members = _members(case, seed)
        graphs = [_host_graph(_dev_graph(f, c, s)) for f, c, s in members]
        opts = B.fw_seg_default_opts(**_opts("knn", case))
        batch = B.Batch(graphs, opts, weight_dtype=case["weights"], lanes_per_row=0)
        return dict(kind=kind, batch=batch, P=len(graphs))
    if kind == "serve":
        members = _members(case, seed)
        reqs = [(_host_graph(_dev_graph(f, c, s)), _opts(f, case)) for f, c, s in members]
        return dict(kind=kind, reqs=reqs,
                    server=_Server(hbm_budget_bytes=2 << 30, max_slots=16, max_K=10,
                                   weight_dtype=case["weights"]))
    family = _FAMILY[kind]
    dev = _dev_graph(family, case, seed)
    if kind == "energy":
        (rp, col, w), lab, K = dev
        n = rp.numel() - 1
        U = torch.rand(n, K, generator=_gen(seed + 1), device=DEV, dtype=torch.float64) ** 3
        U = U / U.sum(1, keepdim=True)
        return dict(kind=kind, rp=rp, col=col, w=w, lab=lab.to(torch.int32), U=U, n=n, K=K,
                    laplacian=case.get("laplacian", "sym"), stream=torch.cuda.current_stream())
    g = _host_graph(dev)
    del dev
    if kind == "newgraph":
        return dict(kind=kind, g=g, opts=_opts(family, case))
    return dict(kind=kind, seg=B.Segmenter(g, **_opts(family, case)))


# --------------------------------------------------------------------- run --

def _stats(*sts):
    """The statistics of one or more solves as a program logs them."""
    return dict(counts=np.array([[st.iters, st.active_rows] for st in sts]),
                values=np.array([[st.gap, st.gap0, st.q, st.alpha, st.objective] for st in sts]))


def run(s):
    kind = s["kind"]
    if kind in ("knn", "sbm", "image"):
        # the handle's graph, solved from its start: statistics, labels and
        # the soft memberships U
        seg = s["seg"]
        seg.reset()
        return dict(stats=_stats(seg.solve()), labels=seg.labels(), U=seg.U())
    if kind == "oneshot":
        return dict(labels=s["seg"].oneshot()[0])
    if kind == "newgraph":
        with B.Segmenter(s["g"], **s["opts"]) as seg:
            return dict(stats=_stats(seg.solve()), labels=seg.labels(), U=seg.U())
    if kind == "batch":
        b = s["batch"]
        b.reset()
        stats = b.solve()
        return dict(stats=_stats(*stats), labels=[b.labels(p) for p in range(s["P"])],
                    U=[b.U(p) for p in range(s["P"])])
    if kind == "serve":
        srv = s["server"]
        tickets = [srv.submit(g, **o) for g, o in s["reqs"]]
        got = [srv.wait(t, g.n) for t, (g, _) in zip(tickets, s["reqs"])]
        return dict(stats=_stats(*[st for _, _, st in got]), labels=[lab for _, lab, _ in got])
    return B.fw_energy_noalloc(s["n"], s["K"], s["rp"].data_ptr(), s["col"].data_ptr(),
                               s["w"].data_ptr(), s["col"].numel(), s["U"].data_ptr(), s["K"],
                               s["lab"].data_ptr(), 50.0, 1000.0, s["laplacian"], s["stream"])


# -------------------------------------------------------------------- work --

def _sizes(case):
    """(rows, classes, estimated entries, weight bytes, column bytes)."""
    w = dict(f32=4, bf16=2, f64=8)[case.get("weights", "f64")]
    kind = case["kind"]
    if kind in ("image", "oneshot", "newgraph") or "width" in case:
        n = case["width"] * case["height"]
        return n, case["K"], 8 * n, w, 2
    if kind in ("sbm", "energy"):
        return case["n"], case["K"], int(case["n"] * case["deg"]), w, 4
    return case["n"], case["K"], 15 * case["n"], w, 2 if case["n"] < 1 << 15 else 4


def _solve_work(n, K, nnz, w, c, t, iters, read_U=True):
    # One iteration reads and writes U and L U and reads the graph; where all
    # of that stays on the chip it comes from HBM once per solve, not once per
    # iteration.  Labels (and U as doubles) leave once.
    per = 4 * t * n * K + (c + w) * nnz + 7 * n
    times = iters if per // 2 > L2_BYTES else 1
    return per * times + 4 * n + (8 * n * K if read_U else 0), iters * (2 * nnz + 12 * n * K)


def work(case):
    kind = case["kind"]
    b = f = 0
    if kind in ("batch", "serve"):
        for fam, c, _ in _members(case, 0):
            n, K, nnz, w, cb = _sizes(dict(kind=fam, weights=case["weights"], **c))
            bb, ff = _solve_work(n, K, nnz, w, cb, 4, case["iters"], kind == "batch")
            if kind == "serve":
                bb += 12 * nnz + 8 * n
            b, f = b + bb, f + ff
        return dict(bytes=b, flops=f)
    n, K, nnz, w, c = _sizes(case)
    if kind == "oneshot":
        return dict(bytes=(c + w) * nnz + 4 * n + 5 * n, flops=2 * nnz * K + 4 * n * K)
    if kind == "energy":
        return dict(bytes=12 * nnz + 8 * n + 8 * n * K, flops=(4 + 2 * K) * nnz + 8 * n * K)
    t = 8 if case["weights"] == "f64" else 4
    b, f = _solve_work(n, K, nnz, w, c, t, case["iters"])
    if kind == "newgraph":
        b += 12 * nnz + 8 * n
    return dict(bytes=b, flops=f)


# ------------------------------------------------------------------- exact --

class _Problem64:
    """The method's quantities in FP64 with plain torch: degrees, L, U_hat."""

    def __init__(self, dev, omega0, laplacian):
        (rp, col, w), lab, K = dev
        n = rp.numel() - 1
        self.n, self.K = n, K
        cnt = (rp[1:] - rp[:-1]).long()
        rows = torch.arange(n, device=DEV).repeat_interleave(cnt)
        one = torch.ones(n, 1, dtype=torch.float64, device=DEV)
        A = torch.sparse_csr_tensor(rp.long(), col.long(), w, (n, n))
        d = (A @ one)[:, 0]
        if laplacian == "comb":
            self.W, self.diag = A, d[:, None]
        else:
            v = w / torch.sqrt(d[rows] * d[col.long()])
            self.W, self.diag = torch.sparse_csr_tensor(rp.long(), col.long(), v, (n, n)), one
        self.om = torch.where(lab >= 0, float(omega0), 0.0).double()[:, None]
        self.hat = torch.full((n, K), 1.0 / K, dtype=torch.float64, device=DEV)
        kept = lab >= 0
        self.hat[kept] = torch.nn.functional.one_hot(lab[kept], K).double()

    def lap(self, X):
        return self.diag * X - self.W @ X

    def energy(self, U, inv_eps):
        return float(0.5 * (U * self.lap(U)).sum() + inv_eps * (U * (1 - U)).sum()
                     + 0.5 * (self.om * (self.hat - U) ** 2).sum())


def _choose(G, U, greedy):
    """Vertex per row (lowest index on ties) and the rows that move."""
    K = U.shape[1]
    binary = ((U == 0) | (U == 1)).all(1)
    M = torch.where(U > 0, G, math.inf) if greedy else G
    ar = torch.arange(K, device=DEV)
    s = torch.where(M == M.min(1, keepdim=True).values, ar, K).min(1).values
    at = binary & (U.gather(1, s[:, None])[:, 0] == 1)
    return s, ~(binary if greedy else at)


def _solve64(dev, o, K):
    P = _Problem64(dev, o["omega0"], o.get("laplacian", "sym"))
    ie = 1.0 / o["eps"]
    greedy = o.get("oracle", "greedy") == "greedy"
    U = P.hat.clone()
    LU = P.lap(U)
    E = P.energy(U, ie)
    it, g0, q, a = 0, None, 0.0, 0.0
    while True:
        G = LU - 2 * ie * U + P.om * (U - P.hat)
        s, moved = _choose(G, U, greedy)
        S = torch.nn.functional.one_hot(s, K).double()
        D = torch.where(moved[:, None], S - U, 0.0)
        Gs = G.gather(1, s[:, None])
        mv = moved[:, None].double()
        LS = P.lap(S)
        q_ = (D * LS).sum() - (D * LU).sum() + (P.om * D * D).sum() - 2 * ie * (D * D).sum()
        g, qn, act = torch.stack([(mv * U * (G - Gs)).sum(), q_, moved.sum().double()]).tolist()
        g0 = g if g0 is None else g0
        tol = o.get("gap_tol", 0.0) * (g0 if o.get("tol_mode") == "rel" else 1.0)
        if act == 0 or g <= tol or it >= o["max_iters"]:
            break
        q, a = qn, 1.0
        if q > 0 and o.get("step_rule", "exact") == "exact":
            a = min(1.0, g / q)
        elif q > 0:
            while a > 2 * (1 - 1e-6) * g / q:
                a *= 0.5
        E = E - a * g + 0.5 * a * a * q
        U = torch.where(moved[:, None], (1 - a) * U + a * S, U)
        LU = (1 - a) * LU + a * LS
        it += 1
    return [g, g0, q, a, E], U.cpu().numpy()


def exact(case, seed):
    """FP64 values of what `run` returns.  Labels, counts and the moved rows
    are whole numbers that follow from rounded values: none for them, except
    the one-shot labels, which are a function of the input alone."""
    kind = case["kind"]
    if kind in ("batch", "serve"):
        got = [_solve64(_dev_graph(fam, c, s), _opts(fam, case), c["K"])
               for fam, c, s in _members(case, seed)]
        out = dict(stats=dict(counts=None, values=np.array([v for v, _ in got])),
                   labels=[None] * len(got))
        if kind == "batch":
            out["U"] = [U for _, U in got]
        return out
    family = _FAMILY[kind]
    dev = _dev_graph(family, case, seed)
    if kind == "energy":
        U = torch.rand(case["n"], case["K"], generator=_gen(seed + 1), device=DEV,
                       dtype=torch.float64) ** 3
        P = _Problem64(dev, 1000.0, case.get("laplacian", "sym"))
        return P.energy(U / U.sum(1, keepdim=True), 1.0 / 50.0)
    o = _opts(family, case)
    if "full" in o.values() or "armijo" in o.values():
        return None    # the steps themselves are whole-number decisions there
    if kind == "oneshot":
        P = _Problem64(dev, o["omega0"], "sym")
        G = P.lap(P.hat) - 2.0 / o["eps"] * P.hat
        s = _choose(G, P.hat, True)[0]
        s = torch.where(dev[1] >= 0, dev[1], s)
        return dict(labels=s.to(torch.int32).cpu().numpy())
    values, U = _solve64(dev, o, case["K"])
    return dict(stats=dict(counts=None, values=np.array([values])), labels=None, U=U)
