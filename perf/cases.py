"""What this library is used for, as cases that can be timed and compared.

Every case is one pass through the public entry points (the binding ``gpm``
and ``learned``) on a seeded random graph, of the sizes that the package's own
workloads, tests and benchmark use:

* ``motif``    gpm_motif_count on a graph in hand: G(n, m), block-model and
               R-MAT graphs, k = 3 .. 6;
* ``clique``   gpm_clique_count / gpm_clique_count_range on a graph in hand:
               power-law (Chung-Lu), R-MAT and block-model graphs;
* ``roots``    gpm_count_roots with per-root sizes over every root (how the
               labels of the learned scheduler are measured);
* ``ingest``   from a host CSR to the counts: gpm_graph_create (validated),
               a clique range, destroy;
* ``batch``    gpm_batch_count on thousands of small graphs;
* ``list``     gpm_list of every clique, the consumer adding up how many
               cliques each vertex is in;
* ``schedule`` the learned scheduler end to end: features, network forward,
               balanced schedule, scheduled count;
* ``train``    one training step of that network: gradient and Adam.
"""
from __future__ import annotations

import base64
import json
import math

import numpy as np
import torch

from paper_2212_04551_gb300 import gpm
from paper_2212_04551_gb300 import graphs as G
from paper_2212_04551_gb300 import learned as L

N_PATTERNS = {3: 2, 4: 6, 5: 21, 6: 112, 7: 853}   # connected patterns of k vertices


def listed():
    return [
        # one call on a small sparse network (the size of bio-diseasome): nothing but latency
        dict(name="motif4_er516", what="motif", graph="er", n=516, m=1200, k=4),
        # the scheduler's training labels: every root's 5-vertex subtree size on a hub-rooted R-MAT graph
        dict(name="roots5_rmat12", what="roots", graph="rmat", scale=12, k=5),
        # an analyst's 4-vertex motif census of a skewed graph of 65,536 vertices
        dict(name="motif4_rmat16", what="motif", graph="rmat", scale=16, k=4),
        # a 5-vertex motif census of a community-structured graph
        dict(name="motif5_sbm2000", what="motif", graph="sbm", n=2000, k=5),
        # one clique size on a large sparse power-law graph: a million light roots, few heavy ones
        dict(name="clique4_chunglu1m", what="clique", graph="chunglu", n=1_000_000, k_lo=4, k_hi=4),
        # every clique size 4 .. 7 of the same graph in one call: the dense core decides
        dict(name="cliques4to7_chunglu1m", what="clique", graph="chunglu", n=1_000_000, k_lo=4, k_hi=7),
        # deep cliques of dense communities
        dict(name="cliques6to12_sbm2000", what="clique", graph="sbm", n=2000, k_lo=6, k_hi=12),
        # a graph that arrives on the host: copy, checks, orientation and the counts
        dict(name="ingest_cliques3to5_rmat16", what="ingest", graph="rmat", scale=16, k_lo=3, k_hi=5),
        # thousands of small graphs (molecules, ego networks), both counts of each
        dict(name="batch4096_cliques4_motifs5", what="batch", graphs=4096, clique_k=4, motif_k=5),
        # listing instead of counting: every 6-clique handed to the host while the kernel runs
        dict(name="list6_sbm2000", what="list", graph="sbm", n=2000, k=6),
        # a census of a skewed graph with the learned schedule, prediction included
        dict(name="schedule_motif4_rmat14", what="schedule", graph="rmat", scale=14, k=4),
        # the scheduler network's training step at its usual minibatch
        dict(name="train4096", what="train", samples=4096),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    what = rng.choice(["motif", "motif", "motif", "clique", "clique", "clique", "roots", "ingest", "batch", "list",
                       "schedule", "train"])
    if what == "motif":
        kind = rng.choice(["er", "sbm", "rmat"])
        if kind == "er":
            n = _log_int(rng, 60, 4000)
            k = rng.choice([3, 4, 5, 6])
            return dict(what=what, graph=kind, n=n, m=int(n * rng.uniform(1.2, 4.0)), k=k)
        if kind == "sbm":
            return dict(what=what, graph=kind, n=rng.randint(150, 2000), k=rng.choice([3, 4, 5]))
        return dict(what=what, graph=kind, scale=rng.randint(8, 16), k=rng.choice([3, 4]))
    if what == "clique":
        kind = rng.choice(["chunglu", "rmat", "sbm"])
        if kind == "chunglu":
            k_lo = rng.randint(3, 5)
            return dict(what=what, graph=kind, n=_log_int(rng, 3000, 950_000), k_lo=k_lo, k_hi=rng.randint(k_lo, 7))
        if kind == "rmat":
            k_lo = rng.randint(3, 5)
            return dict(what=what, graph=kind, scale=rng.randint(9, 16), k_lo=k_lo, k_hi=rng.randint(k_lo, 6))
        k_lo = rng.randint(3, 8)
        return dict(what=what, graph=kind, n=rng.randint(150, 2000), k_lo=k_lo, k_hi=rng.randint(k_lo, 12))
    if what == "roots":
        return dict(what=what, graph="rmat", scale=rng.randint(8, 12), k=rng.choice([4, 5]))
    if what == "ingest":
        k_lo = rng.randint(3, 4)
        return dict(what=what, graph=rng.choice(["rmat", "rmat_any"]), scale=rng.randint(8, 16), k_lo=k_lo,
                    k_hi=rng.randint(k_lo, 5))
    if what == "batch":
        return dict(what=what, graphs=_log_int(rng, 100, 4000), clique_k=rng.choice([0, 3, 4, 5]),
                    motif_k=rng.choice([3, 4, 5]))
    if what == "list":
        return dict(what=what, graph="sbm", n=rng.randint(200, 2000), k=rng.choice([5, 6, 7]))
    if what == "schedule":
        return dict(what=what, graph="rmat", scale=rng.randint(9, 14), k=rng.choice([3, 4]))
    return dict(what=what, samples=_log_int(rng, 65, 8000))


# ---------------------------------------------------------------- inputs

def _pack_edges(n, u, v):
    """(indptr, indices) of the undirected graph with edges u - v, on their device."""
    key = torch.unique(torch.cat([u * n + v, v * n + u]))
    indptr = torch.zeros(n + 1, dtype=torch.int64, device=key.device)
    torch.cumsum(torch.bincount(key // n, minlength=n), 0, out=indptr[1:])
    return indptr.to(torch.int32), (key % n).to(torch.int32)


def _chung_lu(n, seed):
    """graphs.chung_lu's recipe (average degree 16, exponent 2.1, expected
    degrees capped at 20 sqrt(n)), drawn on the GPU: (indptr, indices)."""
    gen = torch.Generator(device="cuda").manual_seed(seed)
    w = (torch.arange(n, dtype=torch.float64, device="cuda") + 1.0) ** (-1.0 / 1.1)
    for _ in range(50):
        w *= 16.0 / w.mean()
        w.clamp_(max=20.0 * math.sqrt(n))
    cdf = torch.cumsum(w / w.sum(), 0)
    ends = torch.rand(2, 8 * n, dtype=torch.float64, device="cuda", generator=gen)
    u, v = torch.searchsorted(cdf, ends).clamp_(max=n - 1)
    keep = u != v
    u, v = u[keep], v[keep]
    return _pack_edges(n, u, v)


def _ba_batch(count, seed):
    """``count`` preferential-attachment graphs (n in 20 .. 400, m_a in 2 .. 6,
    graphs.barabasi_albert's recipe), all grown at once: packed (graph_off,
    indptr, indices) with global ids."""
    rng = np.random.default_rng(seed)
    n = rng.integers(20, 401, count)
    ma = rng.integers(2, 7, count)
    goff = np.zeros(count + 1, dtype=np.int64)
    goff[1:] = np.cumsum(n)
    ends = np.zeros((count, 2 * 6 * 400), dtype=np.int32)     # edge endpoints so far, per graph
    ne = 2 * ma
    us = [np.repeat(ma + goff[:-1], ma)]
    vs = [np.arange(ma.sum()) - np.repeat(np.cumsum(ma) - ma, ma) + np.repeat(goff[:-1], ma)]
    for t in range(6):
        gi = np.nonzero(t < ma)[0]
        ends[gi, 2 * t], ends[gi, 2 * t + 1] = ma[gi], t
    slot = np.arange(6)
    for new in range(3, 400):
        gi = np.nonzero((new > ma) & (new < n))[0]
        used = slot < ma[gi, None]
        picks = np.zeros((gi.size, 6), dtype=np.int64)
        todo = np.arange(gi.size)
        while todo.size:            # rows that picked a vertex twice pick again
            at = (rng.random((todo.size, 6)) * ne[gi[todo], None]).astype(np.int64)
            picks[todo] = np.where(used[todo], ends[gi[todo, None], at], -1 - slot)
            row = np.sort(picks[todo], axis=1)
            todo = todo[(row[:, 1:] == row[:, :-1]).any(axis=1)]
        rows, cols = np.nonzero(used)
        g, p = gi[rows], picks[rows, cols]
        us.append(new + goff[g])
        vs.append(p + goff[g])
        ends[g, ne[g] + 2 * cols], ends[g, ne[g] + 2 * cols + 1] = new, p
        ne[gi] += 2 * ma[gi]
    u, v = (torch.from_numpy(np.concatenate(x)).cuda() for x in (us, vs))
    indptr, indices = _pack_edges(int(goff[-1]), u, v)
    return goff.astype(np.int32), indptr.cpu().numpy(), indices.cpu().numpy()


def _csr(case, seed):
    kind = case["graph"]
    if kind == "er":
        return G.erdos_renyi_m(case["n"], case["m"], seed)
    if kind == "sbm":
        return G.sbm(case["n"], 100, 0.5, 0.01, seed)
    g = G.rmat(case["scale"], 8, 0.57, 0.19, 0.19, seed)
    if kind == "rmat_any":      # vertices in no particular order
        g = G.relabel(g, np.random.default_rng(seed).permutation(g.n))
    return g


def _train_arrays(samples, seed):
    """Features and labels of the scheduler's kind: log1p of heavy-tailed sizes."""
    rng = np.random.default_rng(seed)
    x = np.log1p(np.floor(np.exp(rng.normal(2.0, 1.6, (samples, 8))))).astype(np.float32)
    x[:, 7] = rng.integers(5, 7, samples) / 8.0
    t = (0.9 * x[:, 0] + 0.8 * x[:, 3] + 6.0 * x[:, 7] + rng.normal(0, 0.5, samples)).astype(np.float32)
    return x, t


def prepare(case, seed):
    what = case["what"]
    stream = torch.cuda.current_stream()
    st = dict(what=what, case=case, stream=stream)
    if what == "train":
        x, t = _train_arrays(case["samples"], seed)
        st["x"], st["t"] = torch.from_numpy(x).cuda(), torch.from_numpy(t).cuda()
        st["model"] = L.new_model(seed, stream)
        st["grad"] = torch.zeros(gpm.GPM_MLP_PARAMS, dtype=torch.float32, device="cuda")
        st["loss"] = torch.zeros(1, dtype=torch.float32, device="cuda")
        return st
    if what == "batch":
        goff, indptr, indices = _ba_batch(case["graphs"], seed)
        st["b"] = gpm.gpm_batch_create(goff, indptr, indices, stream=None)
        return st
    if case["graph"] == "chunglu":
        indptr, indices = _chung_lu(case["n"], seed)
        st["g"] = gpm.gpm_graph_create(indptr, indices, case["n"], stream=stream)
        return st
    csr = _csr(case, seed)
    if what == "ingest":
        st["csr"] = csr
        return st
    st["n"] = csr.n
    st["g"] = gpm.graph_from_csr(csr, stream=stream)
    if what == "schedule":
        st["model"], _ = L.load(stream=stream)
    return st


def run(st):
    case, what = st["case"], st["what"]
    if what == "motif":
        return gpm.gpm_motif_count(st["g"], case["k"])
    if what == "clique":
        if case["k_lo"] == case["k_hi"]:
            return gpm.gpm_clique_count(st["g"], case["k_hi"])
        return gpm.gpm_clique_count_range(st["g"], case["k_lo"], case["k_hi"])
    if what == "roots":
        counts, per_root = gpm.gpm_count_roots(st["g"], gpm.GPM_APP_MOTIF, case["k"], None, per_root=True)
        return dict(counts=counts, per_root=per_root)
    if what == "ingest":
        g = gpm.graph_from_csr(st["csr"], stream=st["stream"])
        counts = gpm.gpm_clique_count_range(g, case["k_lo"], case["k_hi"])
        g.close()
        return counts
    if what == "batch":
        cliques, motifs = gpm.gpm_batch_count(st["b"], case["clique_k"], case["motif_k"])
        return [motifs] if cliques is None else [cliques, motifs]
    if what == "list":
        member = np.zeros(st["n"], dtype=np.int64)
        k = case["k"]

        def consumer(records):
            np.add(member, np.bincount(records[:, :k].ravel(), minlength=member.shape[0]), out=member)
            return False

        total = gpm.gpm_list(st["g"], gpm.GPM_APP_CLIQUE, k, consumer)
        return dict(total=total, member=member)
    if what == "schedule":
        g, k = st["g"], case["k"]
        x = L.features(g, st["n"], k)
        score = L.predict(st["model"], x, st["stream"])
        L.schedule(g, gpm.GPM_APP_MOTIF, score)
        counts, _ = gpm.gpm_count_scheduled(g, gpm.GPM_APP_MOTIF, k)
        return dict(x=x, score=score, counts=counts)
    m = st["model"]
    gpm.gpm_mlp_grad(m.w, st["x"], st["t"], st["grad"], st["loss"], st["stream"])
    m.step += 1
    gpm.gpm_mlp_adam(m.master, m.m, m.v, st["grad"], m.step, 3e-3, m.w, st["stream"])
    return dict(loss=st["loss"], grad=st["grad"], master=m.master, m=m.m, v=m.v)


# ------------------------------------------------------- what a pass needs

def work(case):
    """Bytes: the CSR (or the samples and parameters) read once, the results
    written once.  Operations: the network's multiply-adds; counting has no
    arithmetic that it could not do without."""
    what = case["what"]
    p = gpm.GPM_MLP_PARAMS
    if what == "train":
        s = case["samples"]
        return {"bytes": 4 * 9 * s + 2 * p + 4 * 7 * p, "flops": 3 * 2 * s * p}
    if what == "batch":
        n = 210 * case["graphs"]
        m = 4 * n
        return {"bytes": 4 * (n + 2 * m) + 8 * case["graphs"] * ((case["clique_k"] > 0) + N_PATTERNS[case["motif_k"]]),
                "flops": 0}
    kind = case["graph"]
    if kind == "er":
        n, m = case["n"], case["m"]
    elif kind == "sbm":
        n = case["n"]
        m = n * (50 + n // 100) // 2
    elif kind == "chunglu":
        n = case["n"]
        m = int(7.5 * n)
    else:
        n = 1 << case["scale"]
        m = int(7.3 * n)
    out = 8 * n if what == "roots" else 8 * N_PATTERNS[case["k"]] if what == "motif" else 64
    if what == "list":
        out += 8 * n
    flops = 0
    if what == "schedule":
        out += 36 * n
        flops = 2 * p * n
    return {"bytes": 4 * (n + 1 + 2 * m) + out, "flops": flops}


# ------------------------------------------------------------- 64-bit values

def _motif4_exact(csr):
    """The six induced 4-vertex counts (star, path, paw, cycle, diamond,
    clique) from the subgraph counts of the dense adjacency matrix."""
    a = np.zeros((csr.n, csr.n))
    e = csr.edges()
    a[e[:, 0], e[:, 1]] = a[e[:, 1], e[:, 0]] = 1.0
    d = a.sum(1)
    a2 = a @ a
    te = a2[e[:, 0], e[:, 1]]                      # triangles of each edge
    tv = (a2 * a).sum(1) / 2
    tri = tv.sum() / 3
    k4 = sum(a[np.ix_(c, c)].sum() / 2 for c in (np.nonzero(a[u] * a[v])[0] for u, v in e)) / 6
    off = a2 - np.diag(np.diag(a2))
    star = (d * (d - 1) * (d - 2) / 6).sum()
    path = ((d[e[:, 0]] - 1) * (d[e[:, 1]] - 1)).sum() - 3 * tri
    paw = (tv * (d - 2)).sum()
    cyc = (off * (off - 1) / 2).sum() / 4
    dia = (te * (te - 1) / 2).sum()
    i_k4 = k4
    i_dia = dia - 6 * k4
    i_cyc = cyc - dia + 3 * k4
    i_paw = paw - 4 * dia + 12 * k4
    i_path = path - 2 * paw - 4 * cyc + 6 * dia - 12 * k4
    i_star = star - paw + 2 * dia - 4 * k4
    return np.rint([i_star, i_path, i_paw, i_cyc, i_dia, i_k4]).astype(np.uint64)


def _core_numbers(csr):
    """Core number of every vertex, by rounds of removal."""
    deg = csr.degrees().copy()
    src = np.repeat(np.arange(csr.n), np.diff(csr.indptr))
    dst = csr.indices.astype(np.int64)
    core = np.full(csr.n, -1, dtype=np.int64)
    c = 0
    while (core < 0).any():
        gone = (core < 0) & (deg <= c)
        if not gone.any():
            c = int(deg[core < 0].min())
            continue
        core[gone] = c
        hit = gone[src]
        deg -= np.bincount(dst[hit], minlength=csr.n)
        keep = ~hit & ~gone[dst]
        src, dst = src[keep], dst[keep]
    return core


def _features_exact(csr, k):
    n = csr.n
    d = csr.degrees()
    src = np.repeat(np.arange(n), np.diff(csr.indptr))
    dst = csr.indices.astype(np.int64)
    up = (d[src] < d[dst]) | ((d[src] == d[dst]) & (src < dst))
    outdeg = np.bincount(src[up], minlength=n)
    # triangles by their lowest (degree, id) vertex: pairs of out-neighbours that are joined
    tri = np.zeros(n)
    key = src * n + dst                            # sorted: the CSR is
    o, s = dst[up], src[up]
    start = np.concatenate([[0], np.cumsum(outdeg)])
    for lo in range(0, n, 2048):
        hi = min(lo + 2048, n)
        first = np.arange(start[lo], start[hi])
        more = start[s[first] + 1] - first - 1     # later entries of the same list
        a = np.repeat(first, more)
        b = a + 1 + np.arange(a.size) - np.repeat(np.cumsum(more) - more, more)
        want = o[a] * n + o[b]
        at = np.minimum(np.searchsorted(key, want), key.size - 1)
        tri += np.bincount(s[a][key[at] == want], minlength=n)
    x = np.zeros((n, 8))
    x[:, 0] = np.log1p(d)
    x[:, 1] = np.log1p(outdeg)
    x[:, 2] = np.log1p(np.bincount(src[dst > src], minlength=n))
    x[:, 3] = np.log1p(np.bincount(src, weights=d[dst], minlength=n))
    x[:, 4] = np.log1p(np.bincount(src[dst > src], weights=d[dst[dst > src]], minlength=n))
    x[:, 5] = np.log1p(tri)
    x[:, 6] = np.log1p(_core_numbers(csr))
    x[:, 7] = k / 8.0
    return x


def _layers(w):
    cut = np.cumsum([0, 512, 64, 4096, 64, 64, 1])
    w1, b1, w2, b2, w3, b3 = (w[a:b] for a, b in zip(cut, cut[1:]))
    return w1.reshape(64, 8), b1, w2.reshape(64, 64), b2, w3, b3


def _bf16(w):
    return torch.from_numpy(np.ascontiguousarray(w, dtype=np.float32)).bfloat16().double().numpy()


def _train_exact(case, seed):
    x, t = (a.astype(np.float64) for a in _train_arrays(case["samples"], seed))
    # the initial weights, as a user's program draws them: uniform within sqrt(6 / fan_in), zero biases
    rng = np.random.default_rng(seed)
    parts = []
    for bias, shape, fan in ((0, (64, 8), 8), (1, (64,), 0), (0, (64, 64), 64), (1, (64,), 0), (0, (64,), 64), (1, (1,), 0)):
        lim = 0.0 if bias else math.sqrt(6.0 / fan)
        parts.append(np.zeros(shape, np.float32).ravel() if bias else
                     rng.uniform(-lim, lim, size=shape).astype(np.float32).ravel())
    master = np.concatenate(parts).astype(np.float64)
    w1, b1, w2, b2, w3, b3 = _layers(_bf16(master))
    z1 = x @ w1.T + b1
    h1 = np.maximum(z1, 0)
    z2 = h1 @ w2.T + b2
    h2 = np.maximum(z2, 0)
    diff = h2 @ w3 + b3[0] - t
    dy = 2 * diff / t.size
    d2 = np.where(z2 > 0, dy[:, None] * w3, 0)
    d1 = np.where(z1 > 0, d2 @ w2, 0)
    g = np.concatenate([(d1.T @ x).ravel(), d1.sum(0), (d2.T @ h1).ravel(), d2.sum(0), h2.T @ dy, [dy.sum()]])
    mm, vv = 0.1 * g, 0.001 * g * g
    new = master - 3e-3 * (mm / 0.1) / (np.sqrt(vv / 0.001) + 1e-8)
    return dict(loss=np.array([np.mean(diff * diff)]), grad=g, master=new, m=mm, v=vv)


def exact(case, seed):
    what = case["what"]
    if what == "train":
        return _train_exact(case, seed)
    if what == "motif" and case["k"] == 4 and case["graph"] != "rmat" and case["n"] <= 2000:
        return _motif4_exact(_csr(case, seed))
    if what == "schedule":
        csr = _csr(case, seed)
        x = _features_exact(csr, case["k"])
        with open(L.WEIGHTS) as f:
            w = np.frombuffer(base64.b64decode(json.load(f)["master_f32_b64"]), dtype="<f4")
        w1, b1, w2, b2, w3, b3 = _layers(_bf16(w))
        h = np.maximum(np.maximum(x @ w1.T + b1, 0) @ w2.T + b2, 0)
        return dict(x=x, score=h @ w3 + b3[0], counts=None)
    return None
