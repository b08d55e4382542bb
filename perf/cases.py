"""The work a user of this library has it do, as measurable cases.

A case is a dict of plain values; `listed` gives the fixed ones, `draw` more of
the same ranges.  `prepare` makes what a program holds before the call (graph,
states, a context), `run` is one pass through the public entry points and
returns its outputs whole, `work` is the traffic and arithmetic the pass cannot
do without, and `exact` the same outputs from plain numpy / torch in 64 bits.

Kinds of work:
  step      new states on a loaded graph: Algorithm 1 and dPC/dx (autograd)
  estimate  a new graph and states: load, preprocess, Algorithm 1
  states    new states on a loaded graph: sort, Algorithm 2 tables, lambda
  bfs       a new graph, one sigma-counting BFS over it
  msbfs     sigma-counting BFS from up to 512 sources of a loaded graph
  exact     exact percolation centrality (Definition 1) of a loaded graph
  graphs    many uneven graphs in one context: states, Algorithm 1, dPC/dx
"""
import math

import numpy as np
import torch

from paper_2509_11454_gb300 import binding

DEV = "cuda:0"
DELTA = 0.1


def listed():
    return [
        # G(1000, avg degree 8), the smallest documented workload: a training step on a
        # small graph, where launches, synchronisations and host work are all there is
        dict(name="er1000_step", kind="step", family="er", n=1000, param=8, states="uniform", eps=0.05, form="bidir"),
        # Barabasi-Albert 200k, m = 4, x ~ U[0,1]: the documented differentiated workload,
        # an ordinary training step
        dict(name="ba200k_step", kind="step", family="ba", n=200_000, param=4, states="uniform", eps=0.01,
             form="bidir"),
        # directed R-MAT 22, Beta(0.5, 2) states: the benchmark's workload and the largest
        # one, graph and states already in device memory
        dict(name="rmat22_estimate", kind="estimate", family="rmat", n=1 << 22, param=16, states="beta", eps=0.01,
             form="bidir", host=False),
        # the same at scale 20, a size that is no power of two, from pinned host buffers and
        # back: what a caller with data on the host sees end to end
        dict(name="rmat1m_host", kind="estimate", family="rmat", n=1_000_003, param=16, states="beta", eps=0.01,
             form="bidir", host=True),
        # a road-like grid with 5% of its edges deleted: hundreds of small levels, and the
        # vertex-diameter bound of an undirected graph of high diameter
        dict(name="grid90k_estimate", kind="estimate", family="grid", n=300 * 300, param=5, states="uniform", eps=0.02,
             form="bidir", host=False),
        # Barabasi-Albert 100k, m = 5, 10% outbreak, in the library's default (batched) form
        dict(name="ba100k_batched", kind="estimate", family="ba", n=100_000, param=5, states="outbreak", eps=0.01,
             form="batched", host=False),
        # the all-paths estimator (lower variance per sample), a small-world graph
        dict(name="ws20k_allpaths", kind="estimate", family="ws", n=20_000, param=10, states="uniform", eps=0.02,
             form="allpaths", host=False),
        # new states for a loaded graph of ragged size: sort and tables on their own
        dict(name="states1500k", kind="states", n=1_500_007, states="uniform"),
        # a graph is loaded and inspected with one full BFS: validation, in-adjacency, BFS
        dict(name="rmat1m_bfs", kind="bfs", family="rmat", n=1 << 20, param=16),
        # distances and path counts from 200 sources at once
        dict(name="ba100k_msbfs", kind="msbfs", family="ba", n=100_000, param=5, nsrc=200),
        # ground truth on a graph small enough for it
        dict(name="ba3k_exact", kind="exact", family="ba", n=3001, param=4, states="uniform"),
        # a batch of uneven graphs (Watts-Strogatz, Barabasi-Albert, grids) trained together
        dict(name="graphs24_step", kind="graphs", count=24, lo=1000, hi=12_000, eps=0.02, form="bidir"),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["step", "estimate", "estimate", "states", "bfs", "msbfs", "exact", "graphs"])
    st = rng.choice(["uniform", "beta", "outbreak", "seeds"])
    if kind == "step":
        fam, par = rng.choice([("er", 8), ("ba", 3), ("ba", 5), ("ws", 10)])
        return dict(kind=kind, family=fam, n=_log_int(rng, 500, 200_000), param=par,
                    states=rng.choice(["uniform", "beta", "outbreak"]), eps=rng.choice([0.01, 0.02, 0.05]),
                    form="bidir")
    if kind == "estimate":
        form = rng.choice(["bidir", "bidir", "batched", "allpaths"])
        fam, par, hi = {"bidir": rng.choice([("rmat", 16, 4_000_000), ("ba", 4, 300_000), ("grid", 5, 60_000)]),
                        "batched": rng.choice([("ba", 5, 100_000), ("ws", 10, 60_000)]),
                        "allpaths": rng.choice([("ws", 10, 20_000), ("ba", 3, 20_000)])}[form]
        return dict(kind=kind, family=fam, n=_log_int(rng, 1000, hi), param=par, states=st,
                    eps=rng.choice([0.01, 0.02]) if fam != "grid" else 0.02, form=form,
                    host=rng.random() < 0.25)
    if kind == "states":
        return dict(kind=kind, n=_log_int(rng, 1000, 4_000_000), states=st)
    if kind == "bfs":
        fam, par = rng.choice([("rmat", 16), ("ba", 4), ("ws", 10)])
        return dict(kind=kind, family=fam, n=_log_int(rng, 1000, 1_000_000), param=par)
    if kind == "msbfs":
        fam, par = rng.choice([("ba", 5), ("rmat", 16), ("ws", 10)])
        return dict(kind=kind, family=fam, n=_log_int(rng, 1000, 100_000), param=par, nsrc=_log_int(rng, 1, 512))
    if kind == "exact":
        fam, par = rng.choice([("ba", 4), ("er", 8), ("ws", 10), ("rmat", 8)])
        return dict(kind=kind, family=fam, n=_log_int(rng, 100, 4000), param=par, states=st)
    return dict(kind=kind, count=_log_int(rng, 2, 24), lo=rng.choice([500, 1000]), hi=_log_int(rng, 2000, 12_000),
                eps=rng.choice([0.02, 0.05]), form="bidir")


# ------------------------------------------------------------------ inputs
# Seeded on the GPU (a 4M-vertex R-MAT takes well under a second there).

def _gen(seed, salt):
    g = torch.Generator(device=DEV)
    g.manual_seed(1_000_003 * int(seed) + salt)
    return g


def _csr(n, src, dst, undirected):
    """(row_ptr, col) of an edge list: no self-loops or duplicates, rows sorted."""
    if undirected:
        src, dst = torch.cat([src, dst]), torch.cat([dst, src])
    keep = src != dst
    key = torch.unique(src[keep] * n + dst[keep])
    src, dst = key // n, (key % n).to(torch.int32)
    rp = torch.zeros(n + 1, dtype=torch.int64, device=DEV)
    rp[1:] = torch.cumsum(torch.bincount(src, minlength=n), 0)
    return rp, dst


def _graph(family, n, param, seed):
    """(row_ptr, col, directed); param: edges per vertex (er, ba, rmat), lattice degree (ws), deleted percent (grid)."""
    g = _gen(seed, 1)
    if family == "rmat":  # (a, b, c) = (0.57, 0.19, 0.19), ids permuted; ids past n are dropped
        scale = max(1, (n - 1).bit_length())
        m = param * n
        u = torch.zeros(m, dtype=torch.int64, device=DEV)
        v = torch.zeros(m, dtype=torch.int64, device=DEV)
        for bit in range(scale):
            r = torch.rand(m, generator=g, device=DEV)
            u |= (r >= 0.76).to(torch.int64) << bit
            v |= (((r >= 0.57) & (r < 0.76)) | (r >= 0.95)).to(torch.int64) << bit
        perm = torch.randperm(1 << scale, generator=g, device=DEV)
        u, v = perm[u], perm[v]
        keep = (u < n) & (v < n)
        return (*_csr(n, u[keep], v[keep], False), True)
    if family == "er":
        e = torch.randint(0, n, (2, n * param // 2), generator=g, device=DEV)
        return (*_csr(n, e[0], e[1], True), False)
    if family == "ba":
        # every edge's far end copies a uniformly chosen earlier end of the list of ends
        # (preferential attachment); the references are followed to a vertex by doubling
        m = param * n
        i = torch.arange(m, device=DEV)
        ref = (torch.rand(m, generator=g, device=DEV, dtype=torch.float64) * (2 * i + 1)).to(torch.int64)
        ends = torch.empty(2 * m, dtype=torch.int64, device=DEV)
        ends[0::2] = 2 * i
        ends[1::2] = torch.minimum(ref, 2 * i)
        while True:
            nxt = ends[ends]
            if bool((nxt == ends).all()):
                break
            ends = nxt
        return (*_csr(n, i // param, ends[1::2] // 2 // param, True), False)
    if family == "ws":
        half = param // 2
        u = torch.arange(n, device=DEV).repeat_interleave(half)
        v = (u + torch.arange(1, half + 1, device=DEV).repeat(n)) % n
        rew = torch.rand(u.shape[0], generator=g, device=DEV) < 0.05
        v = torch.where(rew, torch.randint(0, n, u.shape, generator=g, device=DEV), v)
        return (*_csr(n, u, v, True), False)
    side = int(math.isqrt(n))
    idx = torch.arange(side * side, device=DEV).view(side, side)
    src = torch.cat([idx[:, :-1].reshape(-1), idx[:-1].reshape(-1)])
    dst = torch.cat([idx[:, 1:].reshape(-1), idx[1:].reshape(-1)])
    keep = torch.rand(src.shape[0], generator=g, device=DEV) >= param / 100.0
    return (*_csr(side * side, src[keep], dst[keep], True), False)


def _states(setting, n, seed):
    g = _gen(seed, 2)
    u = torch.rand(n, generator=g, device=DEV, dtype=torch.float64)
    if setting == "uniform":
        return u
    if setting == "beta":  # Beta(0.5, 2): Gamma(1/2) as z^2/2, Gamma(2) as a sum of two exponentials
        a = torch.randn(n, generator=g, device=DEV, dtype=torch.float64) ** 2 / 2
        w = torch.rand(n, generator=g, device=DEV, dtype=torch.float64)
        return a / (a - torch.log1p(-u) - torch.log1p(-w))
    pick = torch.randperm(n, generator=g, device=DEV)
    x = torch.zeros(n, dtype=torch.float64, device=DEV)
    if setting == "outbreak":  # a random tenth in [0.5, 1], the rest 0
        k = pick[: max(2, n // 10)]
        x[k] = 0.5 + 0.5 * u[k]
    else:  # random seeds at 1, the rest 0
        x[pick[:50]] = 1.0
    return x


def _sizes(case):
    """Vertex counts log-uniform in [lo, hi], the case's own (every seed has graphs of these sizes)."""
    r = np.random.default_rng([case["count"], case["hi"]])
    return np.exp(r.uniform(math.log(case["lo"]), math.log(case["hi"]), case["count"])).astype(np.int64)


def _batch(case, seed):
    """Block-diagonal CSR of the batch's graphs: families in turn."""
    vptr, rps, cols, e = [0], [torch.zeros(1, dtype=torch.int64, device=DEV)], [], 0
    for k, n in enumerate(_sizes(case)):
        fam, par = (("ws", 10), ("ba", 3), ("grid", 5))[k % 3]
        rp, col, _ = _graph(fam, int(n), par, 101 * seed + k)
        rps.append(rp[1:] + e)
        cols.append(col + vptr[-1])
        e += int(col.shape[0])
        vptr.append(vptr[-1] + int(rp.shape[0]) - 1)
    return np.array(vptr, dtype=np.int64), torch.cat(rps), torch.cat(cols)


# ------------------------------------------------------------ prepare, run

def _engine(form):
    opts = {"bidir": dict(form="bidir"), "batched": dict(), "allpaths": dict(estimator="allpaths")}
    return binding.PercIS(0, **opts[form])


def prepare(case, seed):
    kind = case["kind"]
    st = dict(case=case, seed=int(seed))
    if kind == "graphs":
        vptr, rp, col = _batch(case, seed)
        st["eng"] = _engine(case["form"])
        st["eng"].set_options(cuda_graphs=1)
        st["eng"].load_graphs(vptr, rp.cpu().numpy(), col.cpu().numpy())
        n = int(vptr[-1])
    elif kind == "states":  # any graph will do: a sparse random one
        n = case["n"]
        e = torch.randint(0, n, (2, 2 * n), generator=_gen(seed, 4), device=DEV)
        st["eng"] = _engine("bidir")
        st["eng"].load_csr(*_csr(n, e[0], e[1], False), directed=True)
    else:
        rp, col, directed = _graph(case["family"], case["n"], case["param"], seed)
        n = int(rp.shape[0]) - 1
        st["eng"] = _engine(case.get("form", "bidir"))
        if kind in ("step", "msbfs", "exact"):
            st["eng"].load_csr(rp, col, directed=directed)
        else:
            if case.get("host"):
                rp, col = rp.cpu().pin_memory(), col.cpu().pin_memory()
            st.update(rp=rp, col=col, directed=directed)
    if kind == "bfs":
        st["source"] = int(torch.argmax(rp[1:] - rp[:-1]))
    elif kind == "msbfs":
        st["sources"] = torch.randperm(n, generator=_gen(seed, 5), device=DEV)[: case["nsrc"]].cpu().numpy()
    else:
        st["x"] = _states(case.get("states", "uniform"), n, seed)
    if kind in ("step", "graphs"):
        st["grad"] = torch.randn(n, generator=_gen(seed, 6), device=DEV, dtype=torch.float64)
    if kind == "step":
        st["x"].requires_grad_(True)
    elif kind == "exact":
        st["eng"].set_states(st["x"])
    elif kind == "estimate" and case["host"]:
        st["x"] = st["x"].cpu().pin_memory()
        st["out"] = torch.empty(n, dtype=torch.float64).pin_memory()
    return st


def run(state):
    case, eng, seed = state["case"], state["eng"], state["seed"]
    kind = case["kind"]
    if kind == "step":
        pc = binding.percolation_centrality(state["x"], eng, case["eps"], DELTA, seed)
        (gx,) = torch.autograd.grad(pc, state["x"], state["grad"])
        return pc.detach(), gx
    if kind == "estimate":
        eng.load_csr(state["rp"], state["col"], directed=state["directed"])
        eng.set_states(state["x"])
        pc, info = eng.estimate(case["eps"], DELTA, seed, out=state.get("out"))
        return pc, info["ell"]
    if kind == "states":
        eng.set_states(state["x"])
        return eng.prep()
    if kind == "bfs":
        eng.load_csr(state["rp"], state["col"], directed=state["directed"])
        return eng.bfs(state["source"])
    if kind == "msbfs":
        return eng.msbfs(state["sources"])
    if kind == "exact":
        return eng.exact()
    eng.set_states(state["x"])
    pc, infos = eng.estimate_graphs(case["eps"], DELTA, seed)
    return pc, eng.backward(state["grad"]), [f["ell"] for f in infos]


def work(case):
    """Inputs read once, outputs written once; flops: the FP64 operations of Algorithm 2's tables
    and C_v (10 a vertex), of the adjoint (20 a vertex) and of the path counts (one addition an
    edge and source).  Edges are counted before duplicates are merged."""
    kind = case["kind"]
    if kind == "graphs":  # mean size of the log-uniform draw; about 7 CSR entries a vertex
        n = case["count"] * (case["hi"] - case["lo"]) / math.log(case["hi"] / case["lo"])
        return dict(bytes=int(n * (8 + 4 * 7 + 4 * 8)), flops=int(30 * n))
    n = case["n"]
    if kind == "states":  # x in; perm, xs, w, c, r, C_v, lambda out
        return dict(bytes=n * (8 + 4 + 6 * 8), flops=10 * n)
    per = {"rmat": case["param"], "er": case["param"], "ba": 2 * case["param"], "ws": case["param"], "grid": 4}
    nnz = per[case["family"]] * n
    graph = 8 * n + 4 * nnz
    if kind == "step":
        return dict(bytes=graph + 4 * 8 * n, flops=30 * n)
    if kind == "estimate":
        return dict(bytes=graph + 2 * 8 * n, flops=10 * n)
    if kind == "bfs":
        return dict(bytes=graph + 12 * n, flops=nnz)
    if kind == "msbfs":
        return dict(bytes=graph + 12 * n * case["nsrc"], flops=nnz * case["nsrc"])
    return dict(bytes=graph + 2 * 8 * n, flops=5 * nnz * n)


# ------------------------------------------------------------------- exact

def exact(case, seed):
    kind = case["kind"]
    if kind == "states":
        x = _states(case["states"], case["n"], seed).cpu().numpy()
        t = _tables(x)
        return {k: (torch.from_numpy(v) if isinstance(v, np.ndarray) else v) for k, v in t.items()} | dict(
            vertex_diam=case["n"] - 2)
    if kind == "step" and case["n"] <= 2000:
        return _exact_step(case, seed)
    if kind == "bfs":
        rp, col, _ = _graph(case["family"], case["n"], case["param"], seed)
        d, s = _bfs(rp, col, [int(torch.argmax(rp[1:] - rp[:-1]))])
        return d[0], s[0]
    if kind == "msbfs":
        rp, col, _ = _graph(case["family"], case["n"], case["param"], seed)
        src = torch.randperm(case["n"], generator=_gen(seed, 5), device=DEV)[: case["nsrc"]].cpu().tolist()
        return _bfs(rp, col, src)
    if kind == "exact":
        return _exact_centrality(case, seed)
    # the sampled estimates of larger graphs: every sampled path would be replayed in
    # Python, minutes for one pass
    return None


def _tables(x):
    """Sorted states, Algorithm 2's tables (1-based, index n+1 = 0), C_v, lambda, c, d^."""
    n = x.shape[0]
    perm = np.argsort(-x, kind="stable").astype(np.int32)
    xs = x[perm] + 0.0
    i = np.arange(1, n + 1, dtype=np.float64)

    def suffix(a):
        out = np.zeros(n + 2)
        out[1:n + 1] = np.cumsum(a[::-1])[::-1]
        return out

    w = suffix(xs)
    ci = np.zeros(n + 2)
    ci[1:n + 1] = np.maximum(0.0, (n - i + 1) * xs - w[1:n + 1])
    r = suffix(ci[1:n + 1])
    c = float(r[1])
    a = (w[1] - w[1:n + 1]) - (i - 1) * xs + (n - i) * xs - w[2:n + 2]
    Cv = np.empty(n)
    Cv[perm] = c - a
    lam = c / Cv
    return dict(perm=perm, xs=xs, w=w, ci=ci, r=r, Cv=Cv, lam=lam, c=c, dhat=float(lam.max()))


def _bfs(rp, col, sources):
    """Distances (int32, -1 = not reached) and path counts from every source, source-major."""
    n = int(rp.shape[0]) - 1
    dist = torch.full((len(sources), n), -1, dtype=torch.int32, device=DEV)
    sigma = torch.zeros((len(sources), n), dtype=torch.float64, device=DEV)
    tail = torch.repeat_interleave(torch.arange(n, device=DEV), rp[1:] - rp[:-1])
    head = col.to(torch.int64)
    for j0 in range(0, len(sources), 16):
        src = torch.tensor(sources[j0:j0 + 16], device=DEV)
        k = torch.arange(src.shape[0], device=DEV)
        d = torch.full((n, src.shape[0]), -1, dtype=torch.int32, device=DEV)
        s = torch.zeros((n, src.shape[0]), dtype=torch.float64, device=DEV)
        d[src, k], s[src, k] = 0, 1.0
        level = 0
        while True:
            on = torch.where(d == level, s, 0.0)
            live = (on > 0).any(1)[tail]
            add = torch.zeros_like(s).index_add_(0, head[live], on[tail[live]])
            new = (d < 0) & (add > 0)
            if not bool(new.any()):
                break
            level += 1
            d[new] = level
            s[new] = add[new]
        dist[j0:j0 + 16], sigma[j0:j0 + 16] = d.t(), s.t()
    return dist, sigma


def _exact_centrality(case, seed):
    """Definition 1 by Brandes' recurrence with target weights R(x_s - x_w), all sources at once."""
    n = case["n"]
    rp, col, _ = _graph(case["family"], n, case["param"], seed)
    x = _states(case["states"], n, seed)
    dist, sigma = _bfs(rp, col, list(range(n)))
    adj = torch.zeros((n, n), dtype=torch.float64, device=DEV)
    adj[torch.repeat_interleave(torch.arange(n, device=DEV), rp[1:] - rp[:-1]), col.to(torch.int64)] = 1.0
    ramp = torch.clamp(x[:, None] - x[None, :], min=0.0)
    delta = torch.zeros_like(sigma)
    for level in range(int(dist.max()) - 1, -1, -1):
        below = torch.where(dist == level + 1, (ramp + delta) / torch.clamp(sigma, min=1.0), 0.0)
        delta = torch.where(dist == level, sigma * (below @ adj.t()), delta)
    delta.fill_diagonal_(0.0)
    Cv = torch.from_numpy(_tables(x.cpu().numpy())["Cv"]).to(DEV)
    return delta.sum(0) / Cv


def _uniform(seed, i, tag, step):
    """Uniform number in (0, 1] of sample i: Philox4x32-10, counter (i, tag, step // 2)."""
    c, key = [i & 0xffffffff, i >> 32, tag, step >> 1], [seed & 0xffffffff, seed >> 32]
    for _ in range(10):
        p0, p1 = 0xD2511F53 * c[0], 0xCD9E8D57 * c[2]
        c = [(p1 >> 32) ^ c[1] ^ key[0], p1 & 0xffffffff, (p0 >> 32) ^ c[3] ^ key[1], p0 & 0xffffffff]
        key = [(key[0] + 0x9E3779B9) & 0xffffffff, (key[1] + 0xBB67AE85) & 0xffffffff]
    word = (c[3] << 32 | c[2]) if step & 1 else (c[1] << 32 | c[0])
    return ((word >> 11) + 1) * 2.0 ** -53


def _random_path(adj, s, t, draw_u):
    """Internal vertices of one uniform shortest s-t path by the balanced bidirectional BFS; None if there is none."""
    lev, sig, front = [{s: 0}, {t: 0}], [{s: 1}, {t: 1}], [[s], [t]]
    while front[0] and front[1]:
        side = 0 if sum(len(adj[v]) for v in front[0]) <= sum(len(adj[v]) for v in front[1]) else 1
        new = {}
        for u in front[side]:
            for v in adj[u]:
                if v not in lev[side]:
                    new[v] = new.get(v, 0) + sig[side][u]
        d = lev[side][front[side][0]] + 1
        lev[side].update(dict.fromkeys(new, d))
        sig[side].update(new)
        front[side] = list(new)
        meet = sorted(v for v in new if v in lev[1 - side])
        if meet:
            weights = [sig[0][v] * sig[1][v] for v in meet]
            goal, acc = draw_u(0) * sum(weights), 0
            for v, wt in zip(meet, weights):
                acc += wt
                if acc >= goal:
                    break
            path, step = [v], 1
            for z, end in ((0, s), (1, t)):
                cur = v
                while cur != end:
                    goal, acc = draw_u(step) * sig[z][cur], 0
                    for p in adj[cur]:
                        if lev[z].get(p) == lev[z][cur] - 1:
                            acc += sig[z][p]
                            if acc >= goal:
                                break
                    cur, step = p, step + 1
                    path.append(cur)
            return [q for q in path if q != s and q != t]
    return None


def _phase(adj, x, tab, seed, phase, count):
    """Algorithm 2's pairs and their paths: [(s, t, internal vertices)] of the samples with a path, and the lengths."""
    n = x.shape[0]
    perm, xs, w, ci, r, c = (tab[k] for k in ("perm", "xs", "w", "ci", "r", "c"))
    first = (c - r[2:n + 2]) / c
    out, ilen = [], []
    for i in range(count):
        s = int(np.searchsorted(first, _uniform(seed, i, phase, 0))) + 1
        d = np.arange(s, n + 1)
        second = ((d - s + 1) * xs[s - 1] - w[s] + w[d + 1]) / ci[s]
        t = min(n, s + int(np.searchsorted(second, _uniform(seed, i, phase, 1))))
        sv, tv = int(perm[s - 1]), int(perm[t - 1])
        path = _random_path(adj, sv, tv, lambda k: _uniform(seed, i, 2 + phase, k)) if x[sv] > x[tv] else None
        ilen.append(len(path) if path is not None else 0)
        if path is not None:
            out.append((sv, tv, path))
    return out, ilen


def _diameter_bound(adj):
    seen, best = set(), 0
    for root in sorted(range(len(adj)), key=lambda v: (-len(adj[v]), v)):
        if root in seen or not adj[root]:
            continue
        seen.add(root)
        front, ecc = [root], 0
        while True:
            nxt = []
            for u in front:
                for v in adj[u]:
                    if v not in seen:
                        seen.add(v)
                        nxt.append(v)
            if not nxt:
                break
            front, ecc = nxt, ecc + 1
        best = max(best, 2 * ecc - 1)
    return best


def _sample_size(eps, dhat, diam, ilen, p_max):
    """Algorithm 1's second sample size from the first phase (Theorem 1)."""
    l1, tot, sq = len(ilen), sum(ilen), sum(v * v for v in ilen)
    var = (l1 * sq - tot * tot) / (l1 * (l1 - 1))
    lg8, lg4 = math.log(8 / DELTA), math.log(4 / DELTA)
    rho = tot / l1 + math.sqrt(2 * var * lg8 / l1) + 7 * diam * lg8 / (3 * (l1 - 1))
    vhat = dhat * dhat * (p_max + math.sqrt(2 * p_max * lg4 / l1) + lg4 / (3 * l1))
    top = dhat / 2 - math.sqrt(dhat * dhat / 4 - min(dhat * dhat / 4, vhat))

    def f(v):
        gx = v * (dhat - v)
        y = eps * dhat / gx
        return dhat * dhat * math.log(4 * dhat * rho / (v * DELTA)) / (gx * ((1 + y) * math.log(1 + y) - y))

    grid = [top * math.pow(10.0, -12 + 12 * k / 4096) for k in range(4097)]
    best = max(range(4097), key=lambda k: f(grid[k]))
    a, b, val, gr = grid[max(best - 1, 0)], grid[min(best + 1, 4096)], f(grid[best]), (math.sqrt(5) - 1) / 2
    for _ in range(101):
        c1, c2 = b - gr * (b - a), a + gr * (b - a)
        val = max(val, f(c1), f(c2))
        a, b = (a, c2) if f(c1) >= f(c2) else (c1, b)
    return math.ceil(val)


def _exact_step(case, seed):
    """Algorithm 1 with the balanced bidirectional BFS, and the adjoint of its fixed-sample estimate."""
    rp, col, _ = _graph(case["family"], case["n"], case["param"], seed)
    n = int(rp.shape[0]) - 1
    rp, col = rp.cpu().numpy(), col.cpu().numpy()
    adj = [col[rp[v]:rp[v + 1]].tolist() for v in range(n)]
    x = _states(case["states"], n, seed).cpu().numpy()
    g = torch.randn(n, generator=_gen(seed, 6), device=DEV, dtype=torch.float64).cpu().numpy()
    tab = _tables(x)
    lam, Cv, c = tab["lam"], tab["Cv"], tab["c"]

    def counts(samples):
        cnt = np.zeros(n)
        for _, _, path in samples:
            cnt[path] += 1
        return cnt

    l1 = max(1000, math.ceil(math.log(1 / DELTA) / case["eps"]))
    smp, ilen = _phase(adj, x, tab, int(seed), 0, l1)
    ell = _sample_size(case["eps"], tab["dhat"], _diameter_bound(adj), ilen, float((lam * counts(smp)).max() / l1))
    smp, _ = _phase(adj, x, tab, int(seed), 1, ell)
    pc = lam * counts(smp) / ell
    # F_v = (C/l) sum_i a_i(v) R(x_s - x_t) / (R_i C_v): the sampled pairs, then C_v
    grad = np.zeros(n)
    for s, t, path in smp:
        coef = c / ell * float((g[path] / Cv[path]).sum()) / (x[s] - x[t])
        grad[s] += coef
        grad[t] -= coef
    gam = g * pc / Cv
    sign = np.sign(x[:, None] - x[None, :])  # [u, v]: sgn(x_u - x_v)
    rank = sign.sum(1)
    grad -= rank * gam.sum() - sign @ gam - gam * rank
    return torch.from_numpy(pc), torch.from_numpy(grad)
