"""Kernel branches at the sizes where they can go wrong, against the CPU oracle."""
import numpy as np
import pytest

import oracle
from paper_2509_11454_gb300 import synth

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def binding():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2509_11454_gb300 import binding as b

    b.load_library()
    return b


def _engine(binding, g, x=None, **opts):
    eng = binding.PercIS(0)
    if opts:
        eng.set_options(**opts)
    eng.load_csr(g.row_ptr, g.col, directed=g.directed)
    if x is not None:
        eng.set_states(x)
    return eng


def _np(t):
    return t.cpu().numpy()


@pytest.mark.parametrize("side,table_log", [(30, 0), (74, 0), (74, 13), (74, -1)])
def test_bidir_counts_pass_2_53_inside_a_phase(binding, side, table_log):
    """Samples whose counts (or only whose products) pass 2^53 change to FP64
    counts on their own: the others' paths equal the oracle's exactly, theirs
    are shortest paths of the same length (FP64 sums past 2^53 round in the
    order of the additions, so the choice itself may differ there)."""
    g = synth.grid_2d(side, 0.0, 0)
    og = oracle.from_synth(g)
    x = synth.states_uniform(g.n, 1)
    prep = oracle.prepare(x)
    eng = _engine(binding, g, x, form="bidir", bi_table_log=table_log)
    count = 240
    ph = eng.run_phase(3, 1, count)
    ptr, nodes = (_np(v) for v in eng.get_paths(count))
    over = 0
    for i in range(count):
        ref = oracle.run_samples(og, prep, 3, 1, 3, i, 1, keep_paths=True, bidir=True)
        assert int(ph["kind"][i]) == int(ref.kind[0]) and int(ph["ilen"][i]) == int(ref.ilen[0]), i
        path = nodes[ptr[i]:ptr[i + 1]]
        if not ref.overflow:
            assert np.array_equal(path, ref.path_nodes), i
            continue
        over += 1
        rows, cols = np.divmod(np.sort(path), side)  # a monotone staircase between the ends
        s, t = divmod(int(ref.s[0]), side), divmod(int(ref.t[0]), side)
        assert len(set(path.tolist())) == len(path) == abs(s[0] - t[0]) + abs(s[1] - t[1]) - 1, i
        assert rows.min() >= min(s[0], t[0]) and rows.max() <= max(s[0], t[0]), i
        assert cols.min() >= min(s[1], t[1]) and cols.max() <= max(s[1], t[1]), i
    assert (over > 0) == (side > 60) and over < count
    eng.close()


@pytest.mark.parametrize("n,hub", [(2, 0), (65, 0), (300, 129), (513, 128), (700, 400)])
def test_exact_centrality_items(binding, n, hub):
    """Exact centrality where its work splits: one or several words of sources, a last
    batch narrower than the first (n = 513, 700), rows at and above the length a whole
    block shares (128).  Sums of at most n^2 non-negative terms of relative error
    2^-52 each way: 4 n^2 2^-53 relative to the largest value."""
    rng = np.random.default_rng(n)
    src, dst = rng.integers(0, n, 3 * n), rng.integers(0, n, 3 * n)
    src, dst = np.concatenate([src, np.zeros(hub), [0]]), np.concatenate([dst, np.arange(1, hub + 1), [1]])
    g = synth.csr_from_edges(n, src, dst, directed=False)
    x = synth.states_uniform(n, n)
    if n == 2:
        with pytest.raises(RuntimeError):  # C_v = 0: undefined
            _engine(binding, g, x)
        return
    eng = _engine(binding, g, x)
    ref = oracle.exact_pc(oracle.from_synth(g), x)
    assert np.max(np.abs(_np(eng.exact()) - ref)) <= 4 * n * n * 2.0 ** -53 * ref.max()
    eng.close()


@pytest.mark.parametrize("directed", [False, True])
@pytest.mark.parametrize("hub", [31, 1024, 1025, 9000])
def test_plain_bfs_rows_and_levels(binding, directed, hub):
    """The single-source BFS where its work splits: rows of one warp, of a whole
    block's parts (above 1,024 edges, out and in), frontiers one block runs alone
    (a 300-vertex tail, more than one stint) and ones the grid takes; from the hub,
    from the tail's end and truncated at a target; VertexDiamUB."""
    rng = np.random.default_rng(hub)
    n = hub + 2 + 300 + 2000
    a, b = np.arange(2, hub + 2), np.full(hub, 1)
    src = [np.zeros(hub, int), a, np.arange(hub + 2, hub + 302)]
    dst = [a, b, np.arange(hub + 3, hub + 303)]
    src += [[1], rng.integers(hub + 302, n, 6000), [hub + 302]]  # hub 0 -> spokes -> 1 -> tail -> random part
    dst += [[hub + 2], rng.integers(hub + 302, n, 6000), [n - 1]]
    g = synth.csr_from_edges(n, np.concatenate(src), np.concatenate(dst), directed=directed)
    og = oracle.from_synth(g)
    eng = _engine(binding, g)
    for s, t in ((0, -1), (hub + 150, -1), (n - 1, -1), (0, 1), (0, hub + 200), (5, 0), (0, n - 1), (n - 1, n - 2)):
        dist, sigma = (_np(v) for v in eng.bfs(s, t))
        _, rd, rs, _, _, _ = oracle.bfs(og, s, t)
        m = rd >= 0 if t >= 0 else slice(None)  # truncated: the vertices the oracle settled
        assert np.array_equal(dist[m], rd[m]) and np.array_equal(sigma[m], rs[m]), (s, t)
    if not directed:
        assert binding.percis_get_prep(eng.ctx)["vertex_diam"] == oracle.vertex_diam_ub(og)
    eng.close()


@pytest.mark.parametrize("directed", [False, True])
@pytest.mark.parametrize("lanes,direction", [(64, 2), (128, 0), (256, 1), (512, 0), (512, 1)])
def test_batched_rows_and_needed_counts(binding, lanes, direction, directed):
    """The batched form where its work splits: rows around 32, 64 and 256 edges (a
    vertex's eight lanes, a warp, a block), samples whose ancestors alone are counted
    (short levels) and ones counted everywhere (a tail of 40 vertices beyond the levels
    that are safe), against the oracle's one-sided samples."""
    rng = np.random.default_rng(lanes)
    src, dst, n = [], [], 0
    for k in (31, 32, 33, 64, 65, 256, 257, 1500):  # stars, each hub tied to the next star
        src += [np.full(k, n), [n + k], [n + k]]
        dst += [np.arange(n + 1, n + k + 1), [n], [n + k + 1]]
        n += k + 1
    src += [rng.integers(0, n, 6 * n), np.arange(n, n + 40)]
    dst += [rng.integers(0, n, 6 * n), np.arange(n + 1, n + 41)]
    src.append([5])
    dst.append([n])
    n += 41
    g = synth.csr_from_edges(n, np.concatenate(src), np.concatenate(dst), directed=directed)
    x = synth.states_uniform(n, 2)
    og, prep = oracle.from_synth(g), oracle.prepare(x)
    eng = _engine(binding, g, x, lanes=lanes, direction=direction)
    ph = eng.run_phase(7, 1, 400)
    ref = oracle.run_samples(og, prep, 7, 1, 3, 0, 400, keep_paths=False)
    assert not ref.overflow
    for k in ("s", "t", "kind", "ilen", "cnt"):
        assert np.array_equal(_np(ph[k]), getattr(ref, k)), k
    eng.close()


@pytest.mark.parametrize("n,scale", [(2, 1.0), (3, 1.0), (1000, 1.0), (4097, 1e-6), (1000, 1e-300), (500, 1e-318)])
@pytest.mark.parametrize("kind", ["uniform", "ties", "seeds"])
def test_pairs_without_divisions(binding, n, scale, kind):
    """Algorithm 2's searches, whose comparisons divide only next to equality (and always
    where the products leave the normal range): the oracle's pairs."""
    rng = np.random.default_rng(n)
    x = rng.random(n)
    if kind == "ties":
        x = np.round(x * 4) / 4
    elif kind == "seeds":
        x = np.where(x > 0.7, 1.0, 0.0)
    x[: min(n, 3)] = (1.0, 0.5, 0.0)[: min(n, 3)]
    x = x * scale
    g = synth.csr_from_edges(n, np.arange(n), (np.arange(n) + 1) % n, directed=True)
    prep = oracle.prepare(x)
    if not np.all(prep.Cv > 0):
        pytest.skip("undefined states")
    eng = _engine(binding, g, x)
    s, t = eng.sample_pairs(5, 1, 0, 4000)
    rs, rt, _, _ = oracle.sample_pairs(prep, 5, 1, 0, 4000)
    assert np.array_equal(_np(s), rs) and np.array_equal(_np(t), rt)
    eng.close()


@pytest.mark.parametrize("n", [2, 3, 4095, 4096, 4097, 8193, 262144, 262145, 300001])
@pytest.mark.parametrize("kind", ["uniform", "ties", "close", "packed"])
def test_state_sort(binding, n, kind):
    """The states' sort at its tiles, merges and radix passes: ties by vertex id, states
    that agree in their upper 40 bits in short runs (close) and in runs long enough for
    the second sort (packed): the stable order, and the tables that follow from it."""
    rng = np.random.default_rng(n)
    x = rng.random(n)
    if kind == "ties":
        x = np.round(x * 7) / 8
    elif kind == "close":
        x = np.floor(x * (n // 4 + 1)) / (n + 1) + rng.integers(0, 3, n) * 2.0 ** -50
    elif kind == "packed":
        x = 0.5 + rng.integers(0, 1000, n) * 2.0 ** -53
    x[:2] = (1.0, 0.0)
    g = synth.csr_from_edges(n, np.arange(n), (np.arange(n) + 1) % n, directed=True)
    if not np.all(oracle.prepare(x, cv_method="sorted").Cv > 0):  # undefined: reported
        assert n <= 3
        with pytest.raises(RuntimeError, match="C_v <= 0"):
            _engine(binding, g, x)
        return
    eng = _engine(binding, g, x)
    p = eng.prep()
    perm = np.argsort(-x, kind="stable")
    assert np.array_equal(_np(p["perm"]), perm) and np.array_equal(_np(p["xs"]), x[perm])
    w = np.cumsum(x[perm][::-1])[::-1]
    assert np.array_equal(_np(p["w"])[1:n + 1], w)
    eng.close()


@pytest.mark.parametrize("count", [2, 40, 90, 200, 600])
@pytest.mark.parametrize("estimator", ["", "allpaths"])
def test_batches_side_by_side(binding, count, estimator):
    """Batches of 64 lanes from one to more than the groups that run side by side: every
    group's state is its own (counts and paths equal the oracle's; the all-paths sums
    equal those of one batch at a time to the rounding of their additions)."""
    g = synth.barabasi_albert(500, 3, 2)
    x = synth.states_uniform(g.n, 2)
    if estimator:
        est = []
        for instrument in (0, 1):
            eng = _engine(binding, g, x, estimator="allpaths", lanes=64, ell1=count, ell=count, instrument=instrument)
            pc, _ = eng.estimate(0.05, 0.1, 4)
            est.append(_np(pc))
            eng.close()
        # each sum has at most `count` positive terms, in any order: (count - 1) roundings a
        # side, and a few after it
        assert np.all(np.abs(est[0] - est[1]) <= 2 * (count + 4) * 2.0 ** -53 * est[1])
        return
    eng = _engine(binding, g, x, lanes=64)
    ph = eng.run_phase(4, 1, count)
    ptr, nodes = (_np(v) for v in eng.get_paths(count))
    ref = oracle.run_samples(oracle.from_synth(g), oracle.prepare(x), 4, 1, 3, 0, count, keep_paths=True)
    assert np.array_equal(_np(ph["cnt"]), ref.cnt)
    assert np.array_equal(_np(ph["ilen"]), ref.ilen) and np.array_equal(nodes, ref.path_nodes)
    eng.close()


def test_many_graphs_sampling_and_backward_in_one_launch(binding):
    """Path graphs whose samples have up to 2, 7, 8, 9, 16, 17 and 38 internal vertices
    (eight lanes share a sample): pairs, counts and gradients of each graph in the batch
    are the oracle's."""
    sizes = [4, 9, 10, 11, 18, 19, 40]
    graphs = [synth.csr_from_edges(n, np.arange(n - 1), np.arange(1, n), directed=False) for n in sizes]
    vptr, rp, col = synth.union_csr(graphs)
    x = synth.states_uniform(int(vptr[-1]), 3)
    fixed = 300
    eng = binding.PercIS(0)
    eng.set_options(form="bidir", ell1=100, ell=fixed)
    eng.load_graphs(vptr, rp, col)
    eng.set_states(x)
    pc = _np(eng.estimate_graphs(0.05, 0.1, seed=2)[0])
    gvec = np.random.default_rng(3).standard_normal(int(vptr[-1]))
    gx = _np(eng.backward(torch.as_tensor(gvec, device="cuda")))
    for g, graph in enumerate(graphs):
        lo, hi = vptr[g], vptr[g + 1]
        prep = oracle.prepare(x[lo:hi], cv_method="sorted")
        ph = oracle.run_samples(oracle.from_synth(graph), prep, 2, 1, 3, g * fixed, fixed, keep_paths=True, bidir=True)
        F = prep.lam * ph.cnt / fixed
        assert np.max(np.abs(pc[lo:hi] - F)) <= 1e-9, g
        ref = oracle.vjp_fixed(prep, fixed, ph, F, gvec[lo:hi])
        assert np.linalg.norm(gx[lo:hi] - ref) <= 1e-10 * np.linalg.norm(ref), g
    eng.close()


@pytest.mark.parametrize("n", [300, 32768, 32769])
@pytest.mark.parametrize("count", [607, 609, 1300])
def test_bidir_small_graph_blocks(binding, n, count):
    """Samples by 128 threads (graphs of up to 2^15 vertices, more samples than 256-thread
    blocks fit the chip) and by 256: frontiers and meeting layers around a chunk of 256
    vertices (a hub over the whole graph), the oracle's paths."""
    rng = np.random.default_rng(n)
    hub = np.arange(1, min(n, 700))
    src = np.concatenate([np.zeros(len(hub), dtype=np.int64), rng.integers(0, n, 3 * n)])
    dst = np.concatenate([hub, rng.integers(0, n, 3 * n)])
    g = synth.csr_from_edges(n, src, dst, directed=False)
    x = synth.states_uniform(n, 4)
    eng = _engine(binding, g, x, form="bidir")
    ph = eng.run_phase(6, 1, count)
    ptr, nodes = (_np(v) for v in eng.get_paths(count))
    ref = oracle.run_samples(oracle.from_synth(g), oracle.prepare(x), 6, 1, 3, 0, count, keep_paths=True, bidir=True)
    assert not ref.overflow
    for k in ("s", "t", "kind", "ilen", "cnt"):
        assert np.array_equal(_np(ph[k]), getattr(ref, k)), k
    assert np.array_equal(nodes, ref.path_nodes)
    eng.close()


def _csr_with_copies(n, src, dst, copies, directed, rng=None):
    """CSR that keeps every edge as often as it is given (rng: rows in random order)."""
    src, dst = np.repeat(src, copies), np.repeat(dst, copies)
    if not directed:
        src, dst = np.concatenate([src, dst]), np.concatenate([dst, src])
    order = np.lexsort((dst if rng is None else rng.random(len(dst)), src))
    row_ptr = np.concatenate([[0], np.cumsum(np.bincount(src, minlength=n))]).astype(np.int64)
    return synth.Graph(n=n, row_ptr=row_ptr, col=dst[order].astype(np.int32), directed=directed, name="copies")


@pytest.mark.parametrize("directed", [False, True])
@pytest.mark.parametrize("shuffled", [False, True])
@pytest.mark.parametrize("table_log", [0, 10])
@pytest.mark.parametrize("kind", ["path2", "path3", "diamonds", "simple"])
def test_bidir_parallel_edges(binding, kind, table_log, shuffled, directed):
    """Rows that hold a column several times count one path per copy: counts far past 2^53
    (2^199, 3^199, 3^60) on frontiers of one or two vertices.  Every sum has two terms, or
    equal ones, so FP64 counts round alike in any order: pairs, lengths, counts and paths
    are the oracle's exactly, and the flag is raised where the oracle raises it."""
    if kind == "diamonds":  # v -> a, v -> b twice, a -> v', b -> v'
        k = 60
        n, v = 3 * k + 1, 3 * np.arange(k)
        src, dst = np.concatenate([v, v, v + 1, v + 2]), np.concatenate([v + 1, v + 2, v + 3, v + 3])
        copies = np.concatenate([np.ones(k, int), np.full(k, 2), np.ones(2 * k, int)])
    else:
        n = 200
        src, dst = np.arange(n - 1), np.arange(1, n)
        copies = np.full(n - 1, {"path2": 2, "path3": 3, "simple": 1}[kind])
    g = _csr_with_copies(n, src, dst, copies, directed, np.random.default_rng(1) if shuffled else None)
    x = np.linspace(1.0, 0.0, n)
    eng = _engine(binding, g, x, form="bidir", bi_table_log=table_log, ell1=240, ell=240)
    ph = eng.run_phase(3, 1, 240)
    ptr, nodes = (_np(a) for a in eng.get_paths(240))
    ref = oracle.run_samples(oracle.from_synth(g), oracle.prepare(x), 3, 1, 3, 0, 240, keep_paths=True, bidir=True)
    for key in ("s", "t", "kind", "ilen", "cnt"):
        assert np.array_equal(_np(ph[key]), getattr(ref, key)), key
    assert np.array_equal(nodes, ref.path_nodes)
    assert ref.overflow == (kind != "simple")
    assert eng.estimate(0.05, 0.1, 3)[1]["sigma_overflow"] == int(ref.overflow)
    eng.close()


@pytest.mark.parametrize("layers", [[10], [18], [28], [500], [24, 40]])
@pytest.mark.parametrize("scale", [1.0, 1e-300])
def test_exact_centrality_scale_and_counts(binding, layers, scale):
    """Exact centrality where counts are stored in 32 and 64 bits and as FP64 (4^9, 4^17,
    4^27, 4^499 paths over layers of four vertices) and with states of any scale, one
    component's a thousand orders of two below the other's: each value relative to itself.
    A dependency is a sum of non-negative terms over at most `layers` levels, four edges
    and a few roundings each, and a value sums n of them: 2 (8 layers + n) 2^-53."""
    src, dst, xs, lo = [], [], [], 0
    rng = np.random.default_rng(len(layers) + layers[0])
    for c, depth in enumerate(layers):
        at = lo + 4 * np.arange(depth - 1)
        for a in range(4):
            for b in range(4):
                src.append(at + a)
                dst.append(at + 4 + b)
        xs.append(rng.random(4 * depth) * 2.0 ** (-990 * c))
        lo += 4 * depth
    x = np.concatenate(xs) * (scale if len(layers) == 1 else 1.0)
    g = synth.csr_from_edges(lo, np.concatenate(src), np.concatenate(dst), directed=False)
    eng = _engine(binding, g, x)
    ref = oracle.exact_pc(oracle.from_synth(g), x, oracle.prepare(x, cv_method="sorted").Cv)
    got = _np(eng.exact())
    assert np.all(np.abs(got - ref) <= 2 * (8 * max(layers) + lo) * 2.0 ** -53 * ref)
    assert np.count_nonzero(got) > lo // 2
    eng.close()


def _fill(leave):
    """A block of device memory that leaves about `leave` bytes free."""
    torch.cuda.synchronize()
    torch.cuda.empty_cache()
    return torch.empty(torch.cuda.mem_get_info()[0] - leave, dtype=torch.uint8, device="cuda")


def test_batches_side_by_side_in_little_memory(binding):
    """Batches side by side are given up where their memory cannot be had: in a phase that
    fits one batch's state and not two (1.8 GB each), and for a later call that needs what
    they hold.  Counts, paths and distances are those with the memory free."""
    n, count = 1 << 18, 4000
    rng = np.random.default_rng(1)
    src = np.concatenate([np.arange(n), rng.integers(0, n, 2 * n)])
    dst = np.concatenate([(np.arange(n) + 1) % n, rng.integers(0, n, 2 * n)])
    g = synth.csr_from_edges(n, src, dst, directed=False)
    x = synth.states_uniform(n, 1)
    m = 4 * n
    rp2, col2 = np.arange(m + 1, dtype=np.int64) * 4, rng.integers(0, m, 4 * m).astype(np.int32)

    def phase(eng):
        ph = eng.run_phase(7, 1, count)
        return [_np(ph[k]) for k in ("cnt", "ilen")] + [_np(eng.get_paths(count)[1])]

    wide = _engine(binding, g, x, lanes=512)
    free = torch.cuda.mem_get_info()[0]
    ref = phase(wide)
    assert free - torch.cuda.mem_get_info()[0] > 6 << 30  # (four batches)
    filler = _fill(64 << 20)
    wide.load_csr(rp2, col2, directed=True)  # needs more than is free
    dist = _np(wide.bfs(0)[0])
    wide.close()
    del filler
    torch.cuda.empty_cache()
    eng = binding.PercIS(0)
    eng.load_csr(rp2, col2, directed=True)
    assert np.array_equal(_np(eng.bfs(0)[0]), dist)
    eng.close()
    narrow = _engine(binding, g, x, lanes=512)
    filler = _fill(3 << 30)
    for a, b in zip(phase(narrow), ref):
        assert np.array_equal(a, b)
    del filler
    torch.cuda.empty_cache()
    for a, b in zip(phase(narrow), ref):
        assert np.array_equal(a, b)
    narrow.close()


@pytest.mark.parametrize("n,count,leave", [(1 << 18, 400, 7.0), (1 << 18, 400, 2.0), (1 << 15, 1300, 1.6)])
def test_bidir_slots_in_little_memory(binding, n, count, leave):
    """The direct store's slots (14.7 MB each at 2^18 vertices, 608 of them; 1.8 MB and 1,216
    at 2^15) in `leave` GB: as many as can be had, with the same counts and paths."""
    rng = np.random.default_rng(n)
    src, dst = np.arange(n), (np.arange(n) + 1) % n
    src, dst = np.concatenate([src, rng.integers(0, n, 2 * n)]), np.concatenate([dst, rng.integers(0, n, 2 * n)])
    g = synth.csr_from_edges(n, src, dst, directed=False)
    x = synth.states_uniform(n, 1)

    def phase(eng):
        ph = eng.run_phase(7, 1, count)
        return [_np(ph[k]) for k in ("cnt", "ilen")] + [_np(eng.get_paths(count)[1])]

    eng = _engine(binding, g, x, form="bidir", bi_table_log=-1)
    ref = phase(eng)
    eng.close()
    eng = _engine(binding, g, x, form="bidir", bi_table_log=-1)
    filler = _fill(int(leave * 1e9))
    for k in range(2):
        for a, b in zip(phase(eng), ref):
            assert np.array_equal(a, b), k
    del filler
    torch.cuda.empty_cache()
    eng.load_csr(g.row_ptr, g.col)
    eng.set_states(x)
    for a, b in zip(phase(eng), ref):
        assert np.array_equal(a, b)
    eng.close()


def test_phase_after_a_failed_allocation(binding):
    """A phase that runs out of memory leaves no sample and no stale sizes: the path arena
    (2^23 samples with 400 MB free) and the hashed store's tables (5 GB with 1 GB free);
    the phases after it are as ever."""
    g = synth.barabasi_albert(2000, 3, 1)
    x = synth.states_uniform(g.n, 1)
    eng = _engine(binding, g, x, form="bidir")

    def phase():
        ph = eng.run_phase(7, 1, 400)
        return [_np(ph[k]) for k in ("cnt", "ilen")] + [_np(eng.get_paths(400)[1])]

    ref = phase()
    for leave, opts, count in ((400e6, {}, 1 << 23), (1e9, {"bi_table_log": 18, "bi_table_max_log": 18}, 400)):
        eng.set_options(**opts)
        filler = _fill(int(leave))
        with pytest.raises(RuntimeError, match="OOM"):
            binding.percis_run_phase(eng.ctx, 7, 1, count)
        with pytest.raises(RuntimeError, match="NO_SAMPLE"):
            binding.percis_get_paths(eng.ctx)
        del filler
        torch.cuda.empty_cache()
        for a, b in zip(phase(), ref):
            assert np.array_equal(a, b), leave
    eng.close()


@pytest.mark.parametrize("count", [70, 100, 130, 200])
def test_batch_direction_from_its_own_work(binding, count):
    """The work estimates that choose a level's direction are the batch's own: those of the
    last batch (64 lanes, one after the other) before its first level, none, and before its
    second, from the neighbours of its sources."""
    g = synth.barabasi_albert(600, 2, 3)
    eng = _engine(binding, g, synth.states_uniform(g.n, 3), lanes=64, lane_order=0, instrument=1)
    s = _np(eng.run_phase(4, 1, count)["s"])
    rec = binding.percis_last_levels(eng.ctx)
    eng.close()
    u = np.unique(s)
    assert (len(u) > 64) == (count > 70)  # (one batch, or several)
    last = u[(len(u) - 1) // 64 * 64:]
    deg = np.diff(g.row_ptr)
    seen = np.zeros((len(last), g.n), dtype=bool)
    for lane, v in enumerate(last):
        seen[lane, g.col[g.row_ptr[v]:g.row_ptr[v + 1]]] = True
    front = seen.any(axis=0)
    seen[np.arange(len(last)), last] = True
    assert len(rec) >= 2
    assert (rec[0][3], rec[0][1] >> 1) == (0, 0)
    assert (rec[1][3], rec[1][1] >> 1) == (deg[front].sum(), deg[~seen.all(axis=0)].sum())


@pytest.mark.parametrize("n", [3000, 30000, 200000])
def test_plain_bfs_on_a_slightly_larger_graph(binding, n):
    """A graph 1/32 larger than the one the level stamps were allocated for: every vertex of
    a binary tree at its level, also past the first graph's last, where the memory held
    other values before (the states of an engine that has gone)."""
    def tree(n):
        v = np.arange(1, n)
        return synth.csr_from_edges(n, v, (v - 1) // 2, directed=False)

    for _ in range(4):
        old = [_engine(binding, tree(n), 0.5 + 0.5 * synth.states_uniform(n, 1)) for _ in range(4)]
        for eng in old:
            eng.close()
        eng = binding.PercIS(0)
        for k in (n, n + n // 32):
            g = tree(k)
            eng.load_csr(g.row_ptr, g.col)
            dist, sigma = (_np(a) for a in eng.bfs(0))
            assert np.array_equal(dist, np.floor(np.log2(np.arange(k) + 1))) and np.all(sigma == 1), k
        eng.close()


@pytest.mark.parametrize("n,diamond", [(600, False), (200, True)])
@pytest.mark.parametrize("lanes", [64, 512])
def test_batched_needed_counts_past_their_list(binding, n, diamond, lanes):
    """Needed (vertex, level) pairs past the room of their list (2 n; a directed cycle's
    lanes need every vertex at nearly every level, and its walks are too few for the
    counts of all vertices): the counts are then listed level by level; the oracle's."""
    src, dst = np.arange(n), (np.arange(n) + 1) % n
    if diamond:  # 0 -> n -> 2 beside 0 -> 1 -> 2
        src, dst, n = np.append(src, [0, n]), np.append(dst, [n, 2]), n + 1
    g = synth.csr_from_edges(n, src, dst, directed=True)
    x = synth.states_uniform(n, 2)
    eng = _engine(binding, g, x, lanes=lanes)
    ph = eng.run_phase(7, 1, 1500)
    nodes = _np(eng.get_paths(1500)[1])
    ref = oracle.run_samples(oracle.from_synth(g), oracle.prepare(x), 7, 1, 3, 0, 1500, keep_paths=True)
    for k in ("s", "t", "kind", "ilen", "cnt"):
        assert np.array_equal(_np(ph[k]), getattr(ref, k)), k
    assert np.array_equal(nodes, ref.path_nodes) and ref.ilen.sum() > 100 * n
    eng.close()


def test_work_queued_by_torch_is_waited_for(binding):
    """On torch's default stream, beside which the context has a stream of its own: states
    and gradients that are still being made, and an output buffer still being written, are
    waited for (each behind about 10 ms of other work)."""
    g = synth.barabasi_albert(500, 3, 1)
    x = torch.as_tensor(synth.states_uniform(g.n, 1), device="cuda")
    grad = torch.as_tensor(np.random.default_rng(2).standard_normal(g.n), device="cuda")
    eng = _engine(binding, g, x)
    pc = eng.estimate(0.1, 0.1, 3)[0].clone()
    gx = eng.backward(grad).clone()
    torch.cuda.synchronize()

    def late(value):
        buf = torch.full_like(value, 0.25)
        torch.cuda.synchronize()
        torch.cuda._sleep(20_000_000)
        return buf.copy_(value)

    eng.set_states(late(x))
    assert torch.equal(eng.prep()["xs"], torch.sort(x, descending=True).values)
    out = late(x)
    assert torch.equal(eng.estimate(0.1, 0.1, 3, out=out)[0], pc)
    got = eng.backward(late(grad))
    assert torch.linalg.norm(got - gx) <= 1e-10 * torch.linalg.norm(gx)
    eng.close()
