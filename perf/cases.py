"""The calls whose speed is measured, and the 64-bit values they should give.

A case is one call of the package as a user's program makes it: clustering a
point set (with the intermediate results that cluster_detail returns), a
minimum spanning tree alone (single linkage), many independent sets in one
call, the tree stage on a tree the caller already has, or a training step of
the isoperimetric number (forward and backward).  Inputs are made on the GPU
from the seed, with the recipes of paper_1702_04739_gb300/workloads.py
restated in torch so that preparing them is quick.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_1702_04739_gb300 import isoclust

DEV = "cuda"


def listed():
    return [
        # The smallest data set of the method's own evaluation (Wine's shape), as numpy hands it over: a call of latencies.
        dict(name="wine_178x13_f64", kind="cluster", data="blobs", n=178, d=13, k=3, sigma=1.0, dtype="f64", alpha=0.0),
        # The repository's smallest benchmark workload: FP64 blobs.
        dict(name="blobs_2000x8_f64", kind="cluster", data="blobs", n=2000, d=8, k=5, sigma=1.0, dtype="f64", alpha=0.0),
        # Wine Quality's shape with the potential of the outlier mode (alpha > 0).
        dict(name="quality_4898x11_alpha", kind="cluster", data="blobs", n=4898, d=11, k=10, sigma=1.0, dtype="f32",
             alpha=0.01),
        # Internet Ads' shape: few points, long rows; sigma on the scale of the points' spacing.
        dict(name="ads_3279x1558", kind="cluster", data="blobs", n=3279, d=1558, k=2, sigma=40.0, dtype="f32", alpha=0.0),
        # An ordinary FP64 data set from numpy, with a ragged size.
        dict(name="blobs_20011x24_f64", kind="cluster", data="aniso", n=20011, d=24, k=8, sigma=5.0, dtype="f64", alpha=0.0),
        # Single linkage: the spanning tree alone of a middle-sized set, ragged.
        dict(name="mst_30011x20", kind="mst", data="aniso", n=30011, d=20, k=12, dtype="f32"),
        # The benchmark's headline workload: Zipf-sized anisotropic blobs with 2 % outliers.
        dict(name="blobs_100000x64", kind="cluster", data="aniso", n=100000, d=64, k=20, sigma=1.0, dtype="f32", alpha=0.0),
        # Sparse-like L2-normalised feature rows: the largest single set.
        dict(name="sparse_50000x4096", kind="cluster", data="sparse", n=50000, d=4096, k=10, sigma=1.0, dtype="f32", alpha=0.0),
        # A training step of the feature scale: forward and backward of i_k.
        dict(name="train_moons_20000x128", kind="train", data="moons", n=20000, d=128, k=3, sigma=1.0),
        # Thousands of independent sets in one call (the batched workload).
        dict(name="sets_4096_d32", kind="sets", nsets=4096, lo=64, hi=8192, d=32, sigma=1.0),
        # A small ragged batch: a call of latencies again.
        dict(name="sets_32_d8", kind="sets", nsets=32, lo=3, hi=700, d=8, sigma=1.0),
        # The tree stage on a caller's own tree, with potentials.
        dict(name="tree_100000", kind="tree", n=100000, window=1000, k=20),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """One more case of the same ranges."""
    kind = rng.choice(["cluster", "cluster", "cluster_f64", "alpha", "sparse", "mst", "train", "sets", "tree"])
    if kind == "cluster":
        n = _log(rng, 150, 100000)
        d = _log(rng, 2, min(2000, 6.4e11 / (n * n) + 2) if n > 20000 else 1600)
        return dict(kind="cluster", data="aniso" if d <= 256 and n >= 1000 else "blobs", n=n, d=d, k=rng.randint(2, 20),
                    sigma=rng.choice([1.0, round(math.sqrt(d), 2)]), dtype="f32", alpha=0.0)
    if kind == "cluster_f64":
        return dict(kind="cluster", data="blobs", n=_log(rng, 100, 20011), d=_log(rng, 2, 24), k=rng.randint(2, 12),
                    sigma=rng.choice([1.0, 2.5]), dtype="f64", alpha=0.0)
    if kind == "alpha":
        return dict(kind="cluster", data="blobs", n=_log(rng, 200, 10000), d=_log(rng, 2, 40), k=rng.randint(2, 10), sigma=1.0,
                    dtype="f32", alpha=0.01)
    if kind == "sparse":
        n = _log(rng, 1000, 50000)
        return dict(kind="cluster", data="sparse", n=n, d=_log(rng, 500, 4096), k=rng.randint(4, 12), sigma=1.0, dtype="f32",
                    alpha=0.0)
    if kind == "mst":
        return dict(kind="mst", data="aniso", n=_log(rng, 1000, 60000), d=_log(rng, 2, 200), k=rng.randint(4, 20), dtype="f32")
    if kind == "train":
        return dict(kind="train", data="moons", n=_log(rng, 500, 20000), d=_log(rng, 4, 160), k=3, sigma=1.0)
    if kind == "sets":
        return dict(kind="sets", nsets=_log(rng, 8, 1500), lo=rng.choice([3, 64]), hi=_log(rng, 300, 8192), d=_log(rng, 4, 64),
                    sigma=1.0)
    n = _log(rng, 100, 200000)
    return dict(kind="tree", n=n, window=max(1, _log(rng, max(2, n // 300), n)), k=min(n, _log(rng, 1, 500)))


# ------------------------------------------------------------------ inputs
def _randn(g, *shape):
    return torch.randn(*shape, generator=g, device=DEV, dtype=torch.float64)


def _rand(g, *shape):
    return torch.rand(*shape, generator=g, device=DEV, dtype=torch.float64)


def _sizes(weights, total):
    raw = np.asarray(weights, dtype=np.float64) / np.sum(weights) * total
    base = np.floor(raw).astype(np.int64)
    base[np.argsort(-(raw - base), kind="stable")[: int(total - base.sum())]] += 1
    return base


def _points(case, g):
    n, d = case["n"], case["d"]
    k = min(case["k"], n)
    if case["data"] == "blobs":          # equal blobs of unit variance
        which = torch.arange(n, device=DEV) % k
        X = (20.0 * _rand(g, k, d) - 10.0)[which] + _randn(g, n, d)
    elif case["data"] == "aniso":        # rotated blobs of Zipf sizes and 2 % uniform outliers
        out = int(round(0.02 * n))
        parts = []
        for m in _sizes(np.arange(1, k + 1) ** -1.1, n - out):
            Q = torch.linalg.qr(_randn(g, d, d))[0]
            lam = torch.exp(_rand(g, d) * math.log(20.0) + math.log(0.1))
            parts.append(20.0 * _rand(g, d) - 10.0 + (_randn(g, int(m), d) * lam.sqrt()) @ Q.T)
        X = torch.cat(parts)
        lo, hi = X.amin(0), X.amax(0)
        X = torch.cat([X, lo + (hi - lo) * _rand(g, out, d)])
    elif case["data"] == "moons":        # three interleaved arcs embedded in d dimensions, with noise
        m = torch.arange(n, device=DEV) % 3
        t = math.pi * _rand(g, n)
        flip = m == 1
        P = torch.stack([torch.where(flip, 1.0 - t.cos(), m.double() + t.cos()), torch.where(flip, 0.5 - t.sin(), t.sin())], 1)
        Q = torch.linalg.qr(_randn(g, d, d))[0]
        X = P @ Q[:, :2].T + 0.1 * _randn(g, n, d)
    else:                                # sparse-like rows: 1 % of the features, 80 % of them from the group's pool
        pool, nnz = max(1, round(0.05 * d)), max(2, round(0.01 * d))
        which = torch.arange(n, device=DEV) % k
        pools = _rand(g, k, d).argsort(1)[:, :pool]
        inside = pools[which].gather(1, (_rand(g, n, nnz) * pool).long())
        col = torch.where(_rand(g, n, nnz) < 0.8, inside, (_rand(g, n, nnz) * d).long())
        X = torch.zeros(n, d, device=DEV, dtype=torch.float32)
        X.scatter_reduce_(1, col, torch.exp(_randn(g, n, nnz)).float(), "amax")   # (a column drawn twice counts once)
        X /= X.norm(dim=1, keepdim=True)
    X = X[_rand(g, n).argsort()]
    return X.to(torch.float64 if case.get("dtype") == "f64" else torch.float32).contiguous()


def _set_sizes(case):
    rng = np.random.default_rng([case["nsets"], case["lo"], case["hi"], case["d"]])     # a batch's sizes are its shape: not by the seed
    n = np.floor(np.exp(rng.uniform(math.log(case["lo"]), math.log(case["hi"]), case["nsets"]))).astype(np.int64)
    return np.clip(n, case["lo"], case["hi"])


def prepare(case, seed):
    g = torch.Generator(device=DEV)
    g.manual_seed(1000003 * seed + 17)
    st = dict(case)
    if case["kind"] in ("cluster", "mst"):
        st["X"] = _points(case, g)
        st["k"] = min(case["k"], case["n"])
        st["o"] = isoclust.opts(alpha=case["alpha"]) if case.get("alpha") else None
    elif case["kind"] == "train":
        st["X"] = _points(case, g).requires_grad_()
        st["scale"] = (0.8 + 0.45 * _rand(g, case["d"])).requires_grad_()
        st["width"] = torch.tensor(case["sigma"], dtype=torch.float64, device=DEV, requires_grad=True)
    elif case["kind"] == "sets":
        rng = np.random.default_rng(seed)
        sizes = _set_sizes(case)
        ks = np.minimum(rng.integers(2, 9, case["nsets"]), sizes)
        offsets = np.concatenate([[0], np.cumsum(sizes)])
        k_of = torch.from_numpy(np.repeat(ks, sizes)).to(DEV)
        first = torch.from_numpy(np.repeat(8 * np.arange(case["nsets"]), sizes)).to(DEV)
        n = int(offsets[-1])
        blob = first + (torch.arange(n, device=DEV) * 2654435761 >> 7) % k_of
        centres = (20.0 * _rand(g, 8 * case["nsets"], case["d"]) - 10.0).float()
        st["X"] = centres[blob] + torch.randn(n, case["d"], generator=g, device=DEV)
        st["offsets"], st["ks"] = offsets.tolist(), ks.tolist()
    else:
        rng = np.random.default_rng(seed)
        n = case["n"]
        perm = rng.permutation(n)
        idx = np.arange(1, n)
        up = np.maximum(0, idx - 1 - np.floor(rng.random(n - 1) * np.minimum(idx, case["window"])).astype(np.int64))
        parent = np.full(n, -1, dtype=np.int32)
        parent[perm[idx]] = perm[up]
        phi = np.where(parent >= 0, np.exp(-rng.uniform(0.1, 6.0, n)), 0.0)
        host = dict(parent=parent, phi=phi, omega=rng.uniform(0.2, 5.0, n), p=rng.uniform(0.0, 0.3, n))
        st.update({name: torch.from_numpy(a).to(DEV) for name, a in host.items()})
    return st


def run(state):
    kind = state["kind"]
    if kind == "cluster":
        return isoclust.cluster_detail(state["X"], state["k"], state["sigma"], state["o"])
    if kind == "mst":
        return isoclust.cluster_mst(state["X"])
    if kind == "sets":
        return isoclust.cluster_batched(state["X"], state["offsets"], state["ks"], state["sigma"], detail=True)
    if kind == "tree":
        return isoclust.tree_isoperimetric(state["parent"], state["phi"], state["omega"], state["p"], state["k"])
    ik, labels = isoclust.IsoperimetricNumber.apply(state["X"], state["scale"], state["width"], state["k"])
    dX, dscale, dwidth = torch.autograd.grad(ik, (state["X"], state["scale"], state["width"]))
    return dict(i_k=ik.detach(), labels=labels, dX=dX, dscale=dscale, dsigma=dwidth)


def work(case):
    """Each unordered pair of points of a set once: its distance (2 d) and, where omega is asked for, its root,
    exponential and sums (25)."""
    kind = case["kind"]
    if kind == "tree":
        return dict(bytes=case["n"] * (4 + 3 * 8 + 4 + 1) + 8, flops=5 * case["n"])
    if kind == "sets":
        sizes = _set_sizes(case).astype(float)
        n = sizes.sum()
        return dict(bytes=n * (4 * case["d"] + 25) + 16 * case["nsets"], flops=float((sizes * (sizes - 1) / 2).sum()) * (2 * case["d"] + 25))
    n, d = case["n"], case["d"]
    size = 8 if case.get("dtype") == "f64" else 4
    pairs = n * (n - 1) / 2
    if kind == "mst":
        return dict(bytes=n * d * size + 16 * (n - 1), flops=pairs * 2 * d)
    if kind == "train":                  # backward: the pairs with a point in the set of the largest ratio, about a k-th
        return dict(bytes=2 * n * d * size + 4 * n, flops=pairs * (2 * d + 25) + n * n / case["k"] * (4 * d + 30))
    return dict(bytes=n * d * size + n * (5 + 4 + 24) + 16 * (n - 1), flops=pairs * (2 * d + (35 if case["alpha"] else 25)))


# ------------------------------------------------------------------ the same in 64 bits
def _chunks(n, m):
    step = max(1, (1 << 23) // max(1, m))
    return [(i, min(n, i + step)) for i in range(0, n, step)]


def _dist(A, B):
    acc = torch.zeros(A.shape[0], B.shape[0], dtype=torch.float64, device=A.device)
    for t in range(A.shape[1]):
        diff = A[:, t, None] - B[None, :, t]
        acc.addcmul_(diff, diff)
    return acc.sqrt_()


def _weights(X, sigma, alpha):
    n = X.shape[0]
    omega, p = torch.empty(n, dtype=torch.float64, device=X.device), torch.zeros(n, dtype=torch.float64, device=X.device)
    for a, b in _chunks(n, n):
        r = _dist(X[a:b], X)
        r[torch.arange(b - a, device=X.device), torch.arange(a, b, device=X.device)] = 0.0
        if alpha:
            p[a:b] = alpha * r.sum(1)
        w = torch.exp(-r / sigma)
        w[torch.arange(b - a, device=X.device), torch.arange(a, b, device=X.device)] = 0.0
        omega[a:b] = w.sum(1)
    return omega, p


def _prim(X):
    """(parent, d2 of the parent edge) of the spanning tree rooted at point 0 (Prim)."""
    n = X.shape[0]
    best = torch.full((n,), math.inf, dtype=torch.float64, device=X.device)
    src = torch.full((n,), -1, dtype=torch.int64, device=X.device)
    live = torch.ones(n, dtype=torch.bool, device=X.device)
    edge = torch.zeros(n, dtype=torch.float64, device=X.device)
    cur = torch.zeros(1, dtype=torch.int64, device=X.device)
    inf = torch.full_like(best, math.inf)
    for _ in range(n - 1):
        live[cur] = False
        d2 = (X - X[cur]).square_().sum(1)
        closer = (d2 < best) & live
        best = torch.where(closer, d2, best)
        src = torch.where(closer, cur, src)
        cur = torch.where(live, best, inf).argmin().reshape(1)
        edge[cur] = best[cur]
    return src, edge


def _subpartition(parent, phi, omega, p, k):
    """(i_k, beta, label of each vertex) by bisection over the decision walk, leaves first."""
    n = len(parent)
    children = [[] for _ in range(n)]
    root = 0
    for v, u in enumerate(parent):
        if u >= 0:
            children[u].append(v)
        else:
            root = v
    order = [root]
    for v in order:
        order.extend(children[v])
    order.reverse()

    def decide(N, want=False):
        w, q, cuts, mark, top = list(omega), list(p), 0, [-2] * n, 0.0
        for v in order:
            u, e = parent[v], phi[v]
            if u < 0:
                e = 0.0
            lim = N * w[v]
            if e + q[v] <= lim:
                if want:
                    mark[v] = cuts
                    top = max(top, (e + q[v]) / w[v])
                cuts += 1
                if cuts == k:
                    break
                if u >= 0:
                    q[u] += e
            elif q[v] - e < lim:
                if u >= 0:
                    w[u] += w[v]
                    q[u] += q[v]
                    mark[v] = -1
            elif u >= 0:
                q[u] += e
        return (cuts, mark, top) if want else cuts

    lo, hi = 0.0, (sum(phi) + sum(p)) / min(omega) + 1.0
    step = hi
    while decide(step * 2.0 ** -32) >= k and step > 1e-300:
        step *= 2.0 ** -32
    hi, lo = step, step * 2.0 ** -32 if step > 1e-300 else 0.0
    while hi - lo > 4e-16 * hi:
        mid = math.sqrt(lo * hi) if hi > 2.0 * lo > 0.0 else 0.5 * (lo + hi)
        if not lo < mid < hi:
            break
        lo, hi = (lo, mid) if decide(mid) >= k else (mid, hi)
    _, mark, top = decide(hi, True)
    label = [-1] * n
    for v in reversed(order):            # a joined vertex has its parent's set, a cut one its own
        label[v] = mark[v] if mark[v] >= 0 else label[parent[v]] if mark[v] == -1 and parent[v] >= 0 else -1
    return top, hi, label


def _tree(X, Xexact, sigma, alpha, k):
    src, edge = _prim(X)
    phi = torch.exp(-edge.sqrt() / sigma)
    phi[0] = 0.0
    omega, p = _weights(Xexact, sigma, alpha)
    ik, beta, label = _subpartition(src.tolist(), phi.tolist(), omega.tolist(), p.tolist(), k)
    return src, edge, phi, omega, p, ik, beta, label


def _value(x):
    return torch.tensor([x], dtype=torch.float64)


def exact(case, seed):
    st = prepare(case, seed)
    kind = case["kind"]
    if kind == "tree":
        got = _subpartition(*(st[name].tolist() for name in ("parent", "phi", "omega", "p")), case["k"])
        return None, None, _value(got[0])
    if kind == "sets":
        X = st["X"].double()
        off, small = st["offsets"], len(st["X"]) <= 10000
        omega, phi, ik, beta = [], [], [], []
        for b, k in enumerate(st["ks"]):
            S = X[off[b]:off[b + 1]]
            if small:
                _, _, f, om, _, i, be, _ = _tree(S, S, case["sigma"], 0.0, k)
                phi.append(f)
                ik.append(i)
                beta.append(be)
            else:
                om = _weights(S, case["sigma"], 0.0)[0]
            omega.append(om)
        return dict(labels=None, residual=None, i_k=torch.tensor(ik, dtype=torch.float64) if small else None,
                    beta=torch.tensor(beta, dtype=torch.float64) if small else None, parent=None,
                    phi_par=torch.cat(phi) if small else None, omega=torch.cat(omega))
    n, d = case["n"], case["d"]
    if n * n * d > 1e12 or n * n * d > 2e11 and case["data"] == "sparse":
        return None
    if kind == "mst":
        return (None, None, _prim(st["X"].double())[1][1:].sort()[0]) if n <= 60000 else None
    if kind == "cluster":
        X = st["X"].double()
        none = dict.fromkeys(("labels", "residual", "i_k", "parent", "phi_par", "omega", "p", "beta", "edge_u", "edge_v", "edge_d2"))
        if n > 40000:
            return dict(none, omega=_weights(X, case["sigma"], 0.0)[0])
        src, edge, phi, omega, p, ik, beta, _ = _tree(X, X, case["sigma"], case["alpha"], st["k"])
        return dict(none, i_k=_value(ik), phi_par=phi, omega=omega, p=p, beta=_value(beta), edge_d2=edge[1:].sort()[0])
    # a training step: the forward on the scaled points as stored, the derivative through its tree and sets
    X, s, sigma = st["X"].detach().double(), st["scale"].detach(), case["sigma"]
    Z32 = (X * s).float().double()
    src, _, _, _, _, ik, _, label = _tree(Z32, Z32, sigma, 0.0, case["k"])
    Z = X * s
    label = torch.tensor(label, device=DEV)
    child = torch.arange(1, n, device=DEV)
    cut = (Z[child] - Z[src[child]]).square().sum(1).sqrt()
    om32 = _weights(Z32, sigma, 0.0)[0]
    ratio = []
    for j in range(case["k"]):
        edge = (label[child] == j) != (label[src[child]] == j)
        ratio.append(float(torch.exp(-cut[edge] / sigma).sum() / om32[label == j].sum()))
    star = int(np.argmax(ratio))
    inside = label == star
    edge = inside[child] != inside[src[child]]
    v, r = child[edge], cut[edge]
    f = torch.exp(-r / sigma)
    Phi, Phi_s = f.sum(), (f * r).sum() / sigma ** 2
    gphi = torch.zeros_like(Z)
    pull = (-f / (sigma * r))[:, None] * (Z[v] - Z[src[v]])
    gphi.index_add_(0, v, pull)
    gphi.index_add_(0, src[v], -pull)
    A = inside.nonzero()[:, 0]
    gom, Om, Om_s = torch.zeros_like(Z), 0.0, 0.0
    for a, b in _chunks(len(A), n):
        row = torch.arange(b - a, device=DEV)
        r = _dist(Z[A[a:b]], Z)
        r[row, A[a:b]] = 1.0
        w = torch.exp(-r / sigma)
        w[row, A[a:b]] = 0.0
        Om, Om_s = Om + w.sum(), Om_s + (w * r).sum() / sigma ** 2
        c = -w / (sigma * r)
        gom.index_add_(0, A[a:b], c.sum(1)[:, None] * Z[A[a:b]] - c @ Z)
        gom += c.sum(0)[:, None] * Z - c.T @ Z[A[a:b]]
    R = Phi / Om
    dz = (gphi - R * gom) / Om
    return dict(i_k=torch.tensor(ik, dtype=torch.float64), labels=None, dX=dz * s, dscale=(dz * X).sum(0),
                dsigma=(Phi_s - R * Om_s) / Om)
