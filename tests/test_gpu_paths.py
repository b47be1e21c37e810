"""Edges of the kernels' size- and type-dependent paths against the oracle: the
remainders, the smallest and the largest sizes of each, bit-exact (integers, zero
tolerance)."""
import numpy as np
import pytest

import graphgen
import oracle

pytestmark = pytest.mark.gpu


def _buffers(n, k=1):
    import torch
    return [torch.full((k * n,), -7, dtype=torch.int32, device="cuda") for _ in range(2)]


def _comb(spine, teeth):
    """A path whose every vertex carries `teeth` leaves: deep, with rows past a lane's."""
    s = np.arange(spine, dtype=np.int32)
    leaf = np.arange(spine, spine * (1 + teeth), dtype=np.int32)
    return graphgen.EdgeList(spine * (1 + teeth), np.concatenate([s[:-1], np.repeat(s, teeth)]),
                             np.concatenate([s[1:], leaf]))


@pytest.mark.parametrize("layout,cluster", [("csr", 1), ("csr", 0), ("csr", 16), ("dcsc", 1)])
@pytest.mark.parametrize("shape", ["rmat", "comb", "torus", "star", "deep"])
def test_min_parents_of_top_down_levels(gpu_lib, shape, layout, cluster):
    """Minimum-id parents of vertices that the grid, a thread-block cluster and the tiles
    discover top-down: hubs, levels past the byte staging (depth >= 254), rows longer than
    a lane scans, several roots at level 0."""
    bfs = gpu_lib
    e = {"rmat": lambda: graphgen.rmat(13, seed=5), "comb": lambda: _comb(300, 70), "torus": lambda: graphgen.torus(37),
         "star": lambda: graphgen.star(5000), "deep": lambda: graphgen.path(700)}[shape]()
    ref = oracle.build_csr(e.n, e.src, e.dst)
    g = bfs.Graph.from_edges(e.src, e.dst, e.n, dcsc=layout == "dcsc")
    level, parent = _buffers(e.n)
    for mode in (bfs.MODE_DO, bfs.MODE_TD_ONLY):
        o = bfs.options(mode=mode, parent_mode=bfs.PARENT_MIN_ID, cluster_size=cluster,
                        layout=bfs.LAYOUT_DCSC_TILED if layout == "dcsc" else bfs.LAYOUT_CSR)
        for root in graphgen.pick_roots(e, 3, 8).tolist():
            want = oracle.levels(ref, root)
            g.run(root, parent=parent, level=level, opts=o)
            assert np.array_equal(level.cpu().numpy(), want), (mode, root)
            assert np.array_equal(parent.cpu().numpy(), oracle.min_parent(ref, want)), (mode, root)
        roots = graphgen.pick_roots(e, 5, 9).tolist()
        want = np.full(e.n, -1, np.int64)
        for r in roots:
            lv = oracle.levels(ref, r).astype(np.int64)
            want = np.where((want < 0) | ((lv >= 0) & (lv < want)), lv, want)
        g.run_multiroot(roots, parent=parent, level=level, opts=o)
        assert np.array_equal(level.cpu().numpy(), want), mode
        assert np.array_equal(parent.cpu().numpy(), oracle.min_parent(ref, want.astype(np.int32))), mode
    g.close()


@pytest.mark.parametrize("k", [1, 7, 64, 70])
@pytest.mark.parametrize("shape", ["rmat", "star", "hubs", "path14", "path15", "path16", "comb", "er", "deg120"])
def test_multi_rows_and_parents(gpu_lib, shape, k):
    """Batches whose levels end just inside and just past the level planes (depth 14 / 15),
    whose rows are longer than a group pulls before they become tasks, that do not fill
    their lanes, with both row orders and both directions alone."""
    bfs = gpu_lib
    rng = np.random.default_rng(3)
    e = {"rmat": lambda: graphgen.rmat(12, seed=6), "star": lambda: graphgen.star(4001),
         # two hubs that share 3000 leaves, ids scattered: long rows with late hits
         "hubs": lambda: graphgen.EdgeList(3002, np.repeat(np.array([17, 2900], np.int32), 3002),
                                           np.tile(rng.permutation(3002).astype(np.int32), 2)),
         "path14": lambda: graphgen.path(15), "path15": lambda: graphgen.path(16), "path16": lambda: graphgen.path(17),
         # more rows past a group's steps than the list of chunk tasks holds
         "deg120": lambda: graphgen.erdos_renyi(6000, 360_000, seed=7),
         "comb": lambda: _comb(40, 300), "er": lambda: graphgen.erdos_renyi(3333, 9000, seed=2)}[shape]()
    ref = oracle.build_csr(e.n, e.src, e.dst)
    g = bfs.Graph.from_edges(e.src, e.dst, e.n, hub_first=True)
    roots = rng.choice(graphgen.pick_roots(e, 64, 5), k).tolist()
    want = np.stack([oracle.levels(ref, r) for r in roots])
    pmin = np.stack([oracle.min_parent(ref, w) for w in want])
    level, parent = _buffers(e.n, k)
    for mode in (bfs.MODE_DO, bfs.MODE_TD_ONLY, bfs.MODE_BU_ONLY):
        for rows in (bfs.BU_ROWS_BY_ID, bfs.BU_ROWS_HUB_FIRST):
            level.fill_(-7)
            parent.fill_(-7)
            g.run_multi(roots, level, parent=parent, opts=bfs.options(mode=mode, bu_rows=rows))
            g.sync()
            assert np.array_equal(level.cpu().numpy().reshape(k, e.n), want), (mode, rows)
            assert np.array_equal(parent.cpu().numpy().reshape(k, e.n), pmin), (mode, rows)
    g.close()


@pytest.mark.parametrize("n", [1, 31, 33, 4096, 4097, 40_000, 155_649, 320_001])
@pytest.mark.parametrize("hub", [False, True])
def test_bottom_up_chunk_widths(gpu_lib, n, hub):
    """Bottom-up sweeps whose warps take 1 to 32 bitmap words each (the width follows the
    bitmap's size), with a ragged last word: levels, parents and the searchers' counts."""
    bfs = gpu_lib
    e = graphgen.erdos_renyi(n, 4 * n, seed=n) if n > 1 else graphgen.from_pairs(1, [(0, 0)])
    ref = oracle.build_csr(e.n, e.src, e.dst)
    scan = oracle.hub_first(ref) if hub else ref
    labels = oracle.components(ref)
    g = bfs.Graph.from_edges(e.src, e.dst, e.n, hub_first=hub)
    level, parent = _buffers(e.n)
    rows = bfs.BU_ROWS_HUB_FIRST if hub else bfs.BU_ROWS_BY_ID
    for root in ([0, n // 2] if n > 1 else [0]):
        want = oracle.levels(ref, root)
        for mode, omode in ((bfs.MODE_BU_ONLY, oracle.MODE_BU), (bfs.MODE_DO, oracle.MODE_DO)):
            info = g.run(root, parent=parent, level=level, opts=bfs.options(mode=mode, bu_rows=rows), stats=True,
                         record_levels=256)
            lv = level.cpu().numpy()
            assert np.array_equal(lv, want), (root, mode)
            assert oracle.certify(ref, root, lv, parent.cpu().numpy(), labels) == (0, -1), (root, mode)
            s = oracle.do_schedule(scan, want, omode)
            for col, name in enumerate(["dir", "nf", "mf", "nnext", "mnext", "scanned", "examined"]):
                assert np.array_equal(info["records"][:, col], getattr(s, name)), (root, mode, name)
    g.close()


@pytest.mark.parametrize("shape", ["er", "hubs"])
def test_large_graph_outputs(gpu_lib, shape):
    """Graphs whose parent array exceeds what stays in L2 (top-down levels then take their
    targets by windows), with a ragged last block: claims from short rows and from hubs,
    first windows, row heads and long rows; both row orders, every direction, several
    roots, with and without levels."""
    import torch
    bfs = gpu_lib
    n = (1 << 23) + 77
    if shape == "er":
        e = graphgen.erdos_renyi(n, 3 * n, seed=4)
    else:
        # 40 hubs over overlapping slices of the ids, and a sparse random rest
        rng = np.random.default_rng(5)
        ids = rng.permutation(n).astype(np.int32)
        cut = [ids[i * 150_000:i * 150_000 + 400_000] for i in range(40)]
        r = graphgen.erdos_renyi(n, n, seed=6)
        e = graphgen.EdgeList(n, np.concatenate([np.full(400_000, ids[i], np.int32) for i in range(40)] + [r.src]),
                              np.concatenate(cut + [r.dst]))
    ref = oracle.build_csr(e.n, e.src, e.dst)
    labels = oracle.components(ref)
    g = bfs.Graph.from_edges(e.src, e.dst, e.n, hub_first=True)
    level, parent = _buffers(n)
    root = int(graphgen.pick_roots(e, 1, 3)[0])
    want = oracle.levels(ref, root)
    for mode in (bfs.MODE_DO, bfs.MODE_TD_ONLY, bfs.MODE_BU_ONLY):
        for rows in (bfs.BU_ROWS_BY_ID, bfs.BU_ROWS_HUB_FIRST):
            o = bfs.options(mode=mode, bu_rows=rows)
            parent.fill_(-7)
            g.run(root, parent=parent, level=level, opts=o)
            assert np.array_equal(level.cpu().numpy(), want), (mode, rows)
            assert oracle.certify(ref, root, want, parent.cpu().numpy(), labels) == (0, -1), (mode, rows)
            parent.fill_(-7)
            g.run(root, parent=parent, opts=o)
            assert oracle.certify(ref, root, want, parent.cpu().numpy(), labels) == (0, -1), (mode, rows, "no levels")
    # an output that starts off a 16-byte boundary
    off = torch.full((n + 1,), -7, dtype=torch.int32, device="cuda")
    g.run(root, parent=off[1:], level=level)
    assert oracle.certify(ref, root, want, off[1:].cpu().numpy(), labels) == (0, -1)
    # several roots: every root its own parent, every other vertex one level below its parent
    roots = np.unique(graphgen.pick_roots(e, 9, 4))
    g.run_multiroot(roots, parent=parent, level=level)
    lv, pa = level.cpu().numpy(), parent.cpu().numpy()
    assert (lv[roots] == 0).all() and (pa[roots] == roots).all()
    v = np.flatnonzero(lv > 0)
    assert np.array_equal(lv[pa[v]], lv[v] - 1) and np.array_equal(pa < 0, lv < 0)
    for x in v[:: max(1, v.size // 2000)]:
        assert pa[x] in ref.cols[ref.offsets[x]:ref.offsets[x + 1]]
    g.close()


@pytest.mark.parametrize("big,chunk", [(0, 0), (64, 64), (64, 4096), (300, 200)])
def test_hub_slices_at_class_edges(gpu_lib, big, chunk):
    """Top-down rows shared by all warps: degrees just below and at every class of slice
    counts (1, 4, 16, 64, 256 chunks), alone and many of a class, over overlapping
    targets."""
    bfs = gpu_lib
    n = 60_000
    c = chunk or 128
    degs = sorted({int(max(1, min(n // 2, d))) for k in (1, 4, 16, 64, 256) for d in
                   (c * (k - 1), c * (k - 1) + 1, c * k, c * k + 1)} | {big or 96, (big or 96) + 1} | {70 + i for i in range(40)})
    rng = np.random.default_rng(big + chunk)
    hubs = np.arange(1, 1 + len(degs), dtype=np.int32)
    src, dst = [np.zeros(len(degs), np.int32)], [hubs]
    for h, d in zip(hubs, degs):
        t = rng.choice(np.arange(1 + len(degs), n, dtype=np.int32), d, replace=False)
        src.append(np.full(d, h, np.int32))
        dst.append(t)
    perm = rng.permutation(n).astype(np.int32)
    e = graphgen.EdgeList(n, perm[np.concatenate(src)], perm[np.concatenate(dst)])
    ref = oracle.build_csr(e.n, e.src, e.dst)
    labels = oracle.components(ref)
    g = bfs.Graph.from_edges(e.src, e.dst, e.n)
    level, parent = _buffers(n)
    root = int(perm[0])
    want = oracle.levels(ref, root)
    s = oracle.do_schedule(ref, want, oracle.MODE_TD)
    for pm in (bfs.PARENT_ANY, bfs.PARENT_MIN_ID):
        info = g.run(root, parent=parent, level=level, stats=True, record_levels=64,
                     opts=bfs.options(mode=bfs.MODE_TD_ONLY, parent_mode=pm, td_big_degree=big, td_chunk=chunk))
        pa = parent.cpu().numpy()
        assert np.array_equal(level.cpu().numpy(), want)
        assert oracle.certify(ref, root, want, pa, labels) == (0, -1)
        assert pm == bfs.PARENT_ANY or np.array_equal(pa, oracle.min_parent(ref, want))
        for col, name in enumerate(["dir", "nf", "mf", "nnext", "mnext"]):
            assert np.array_equal(info["records"][:, col], getattr(s, name)), name
    g.close()


@pytest.mark.parametrize("shape", ["hub", "er", "tiny", "union"])
@pytest.mark.parametrize("min_id", [False, True])
def test_dcsc_streams_and_long_columns(gpu_lib, shape, min_id):
    """Tiles whose columns run past a lane's, a group's and a warp's share of them, tiles of
    several units, empty tiles, frontiers on both sides of the streaming rule."""
    bfs = gpu_lib
    rng = np.random.default_rng(11)
    if shape == "hub":
        n = 20_000
        h = rng.integers(0, n, 6)
        e = graphgen.EdgeList(n, np.concatenate([np.repeat(h, 9000), rng.integers(0, n, 30_000)]).astype(np.int32),
                              np.concatenate([rng.integers(0, n, 54_000), rng.integers(0, n, 30_000)]).astype(np.int32))
    elif shape == "er":
        e = graphgen.erdos_renyi(150_001, 1_500_000, seed=3)
    elif shape == "tiny":
        e = graphgen.random_small(65, 400, 2)
    else:
        e, _ = graphgen.disjoint_union([graphgen.complete(60), graphgen.path(9000), graphgen.star(3000)])
    ref = oracle.build_csr(e.n, e.src, e.dst)
    labels = oracle.components(ref)
    g = bfs.Graph.from_edges(e.src, e.dst, e.n, dcsc=True)
    level, parent = _buffers(e.n)
    for root in graphgen.pick_roots(e, 3, 1).tolist():
        want = oracle.levels(ref, root)
        for mode in (bfs.MODE_DO, bfs.MODE_TD_ONLY, bfs.MODE_BU_ONLY):
            if mode == bfs.MODE_BU_ONLY and want.max() > 2000:
                continue
            g.run(root, parent=parent, level=level,
                  opts=bfs.options(mode=mode, layout=bfs.LAYOUT_DCSC_TILED,
                                   parent_mode=bfs.PARENT_MIN_ID if min_id else bfs.PARENT_ANY))
            pa = parent.cpu().numpy()
            assert np.array_equal(level.cpu().numpy(), want), (root, mode)
            assert oracle.certify(ref, root, want, pa, labels) == (0, -1), (root, mode)
            assert not min_id or np.array_equal(pa, oracle.min_parent(ref, want)), (root, mode)
    g.close()


def _mesh(w, h, diag, seed):
    """A w x h grid without wrap-around (degree <= 4; <= 8 with `diag`), ids shuffled."""
    ids = np.random.default_rng(seed).permutation(w * h).astype(np.int32).reshape(h, w)
    pairs = [(ids[:, :-1], ids[:, 1:]), (ids[:-1], ids[1:])]
    if diag:
        pairs += [(ids[:-1, :-1], ids[1:, 1:]), (ids[:-1, 1:], ids[1:, :-1])]
    return graphgen.EdgeList(w * h, np.concatenate([a.ravel() for a, _ in pairs]),
                             np.concatenate([b.ravel() for _, b in pairs]))


@pytest.mark.parametrize("shape", ["mesh4", "mesh8", "narrow", "tree", "path"])
@pytest.mark.parametrize("min_id", [False, True])
def test_cluster_levels_of_short_rows(gpu_lib, shape, min_id):
    """Cluster levels with 4 and 8 lanes per entry and past them: frontiers from one vertex to
    more than a CTA's even share, uneven shares, frontiers that outgrow the cluster (a
    binary tree doubles to the grid's), depths past the byte staging, several roots."""
    bfs = gpu_lib
    rng = np.random.default_rng(4)
    if shape == "tree":
        n = (1 << 15) - 1
        ids = rng.permutation(n).astype(np.int32)
        e = graphgen.EdgeList(n, ids[(np.arange(1, n) - 1) // 2], ids[1:])
    else:
        e = {"mesh4": lambda: _mesh(300, 210, False, 1), "mesh8": lambda: _mesh(180, 190, True, 2),
             "narrow": lambda: _mesh(3, 900, True, 3), "path": lambda: graphgen.path(600)}[shape]()
    ref = oracle.build_csr(e.n, e.src, e.dst)
    labels = oracle.components(ref)
    g = bfs.Graph.from_edges(e.src, e.dst, e.n)
    level, parent = _buffers(e.n)
    pm = bfs.PARENT_MIN_ID if min_id else bfs.PARENT_ANY
    for root in graphgen.pick_roots(e, 3, 6).tolist():
        want = oracle.levels(ref, root)
        for mode, omode in ((bfs.MODE_DO, oracle.MODE_DO), (bfs.MODE_TD_ONLY, oracle.MODE_TD)):
            for c in (0, 2, 8):
                parent.fill_(-7)
                info = g.run(root, parent=parent, level=level, stats=True, record_levels=2048,
                             opts=bfs.options(mode=mode, parent_mode=pm, cluster_size=c))
                pa = parent.cpu().numpy()
                assert np.array_equal(level.cpu().numpy(), want), (root, mode, c)
                assert oracle.certify(ref, root, want, pa, labels) == (0, -1), (root, mode, c)
                assert not min_id or np.array_equal(pa, oracle.min_parent(ref, want)), (root, mode, c)
                s = oracle.do_schedule(ref, want, omode)
                for col, name in enumerate(["dir", "nf", "mf", "nnext", "mnext", "scanned", "examined"]):
                    assert np.array_equal(info["records"][:, col], getattr(s, name)), (root, mode, c, name)
                assert (np.diff(info["records"][:, 7]) >= 0).all()
    roots = np.unique(graphgen.pick_roots(e, 40, 7))
    g.run_multiroot(roots, parent=parent, level=level, opts=bfs.options(parent_mode=pm))
    lv, pa = level.cpu().numpy(), parent.cpu().numpy()
    want = np.min(np.stack([np.where(x < 0, 1 << 30, x) for x in (oracle.levels(ref, int(r)) for r in roots)]), axis=0)
    assert np.array_equal(lv, np.where(want == 1 << 30, -1, want))
    v = np.flatnonzero(lv > 0)
    assert np.array_equal(lv[pa[v]], lv[v] - 1) and np.array_equal(pa[roots], roots)
    g.close()


@pytest.mark.parametrize("chunk", [64, 128, 4096])
def test_hub_slices_by_windows(gpu_lib, chunk):
    """A graph of 2^25 vertices and some, whose heavy rows are taken by windows of the
    targets: degrees at every class of slice counts below, at and above the 64 windows.
    One root, the hubs, their targets: levels, smallest parents and counts are known."""
    bfs = gpu_lib
    n = (1 << 25) + 3
    degs = [d for k in (1, 4, 16, 64, 256, 1024) for d in (chunk * (k - 1) + 1, chunk * k, chunk * k + 1)]
    degs = [d for d in degs if d < n // 16] + [97] * 70 + [4 * chunk + 5] * 70
    rng = np.random.default_rng(chunk)
    ids = rng.permutation(n).astype(np.int32)
    root, hubs, rest = ids[0], ids[1:1 + len(degs)], ids[1 + len(degs):]
    src, dst = [np.full(hubs.size, root)], [hubs]
    for h, d in zip(hubs, degs):
        src.append(np.full(d, h))
        dst.append(rng.choice(rest[:2_000_000] if d < 1000 else rest, d, replace=False) if d < 100_000 else
                   rest[rng.integers(0, rest.size - d):][:d])
    want_parent = np.full(n, n, np.int32)
    for s, t in zip(src, dst):
        np.minimum.at(want_parent, t, s)
    level = np.where(want_parent < n, 2, -1).astype(np.int32)
    level[hubs], level[root] = 1, 0
    want_parent[want_parent == n] = -1
    want_parent[root], want_parent[hubs] = root, root
    g = bfs.Graph.from_edges(np.concatenate(src), np.concatenate(dst), n)
    lv, pa = _buffers(n)
    edges = sum(degs)
    for pm in (bfs.PARENT_ANY, bfs.PARENT_MIN_ID):
        info = g.run(int(root), parent=pa, level=lv, stats=True, record_levels=8,
                     opts=bfs.options(mode=bfs.MODE_TD_ONLY, parent_mode=pm, td_chunk=chunk))
        assert np.array_equal(lv.cpu().numpy(), level)
        p = pa.cpu().numpy()
        two = np.flatnonzero(level == 2)
        assert (level[p[two]] == 1).all() and np.array_equal(p < 0, level < 0)
        if pm == bfs.PARENT_MIN_ID:
            assert np.array_equal(p, want_parent)
        else:   # each parent is a hub with that edge
            key = np.sort(np.concatenate([np.full(t.size, s, np.int64) * n + t for s, t in zip(src[1:], dst[1:])]))
            k = p[two].astype(np.int64) * n + two
            assert (key[np.searchsorted(key, k)] == k).all()
        assert info["records"][1, 2] == edges + hubs.size and info["records"][1, 3] == two.size
        assert info["records"][1, 8] == sum(-(-(d + 1) // chunk) for d in degs if d + 1 > 96)   # chunks of heavy rows
    g.close()


def test_multi_without_room_for_planes(gpu_lib, monkeypatch):
    """The batched search where the allocator refuses the level planes."""
    import torch
    bfs = gpu_lib
    e = graphgen.rmat(12, seed=6)
    ref = oracle.build_csr(e.n, e.src, e.dst)
    g = bfs.Graph.from_edges(e.src, e.dst, e.n)
    roots = [int(r) for r in graphgen.pick_roots(e, 40, 5)]
    level, parent = _buffers(e.n, len(roots))
    alloc, refused = torch.cuda.caching_allocator_alloc, []

    def short_of_memory(nbytes, *rest):
        if nbytes == 32 * e.n:
            refused.append(nbytes)
            raise torch.cuda.OutOfMemoryError("no room")
        return alloc(nbytes, *rest)

    monkeypatch.setattr(torch.cuda, "caching_allocator_alloc", short_of_memory)
    g.run_multi(roots, level, parent=parent)
    g.sync()
    assert refused
    want = [oracle.levels(ref, r) for r in roots]
    assert np.array_equal(level.cpu().numpy().reshape(-1, e.n), np.stack(want))
    assert np.array_equal(parent.cpu().numpy().reshape(-1, e.n), np.stack([oracle.min_parent(ref, w) for w in want]))
    g.close()


@pytest.mark.parametrize("min_id", [False, True])
@pytest.mark.parametrize("cluster", [2, 16])
def test_cluster_episodes_of_one_level(gpu_lib, cluster, min_id):
    """Cluster episodes that end at once, after which the other CTAs may still be on their
    way out of the barrier before: components of a few vertices (the search ends in the
    episode that starts it) and chains of brooms (a path, then a fan that outgrows the
    cluster, again and again: the grid and the cluster take turns, from every counter slot),
    one search right behind the other and from several roots."""
    import torch
    bfs = gpu_lib
    src, dst, n = [], [], 0
    tiny = []
    for k in range(60):            # an edge, a path of three, a star of 20
        tiny.append(n)
        for a, b in ([(0, 1)], [(0, 1), (1, 2)], [(0, j) for j in range(1, 21)])[k % 3]:
            src.append([n + a]); dst.append([n + b])
        n += (2, 3, 21)[k % 3]
    start = n
    for j in range(7):             # handle of j % 4 + 1 vertices, then 100 x 100 leaves, then the next
        h = np.arange(n, n + j % 4 + 2)
        src.append(h[:-1]); dst.append(h[1:])
        mid = np.arange(h[-1] + 1, h[-1] + 101)
        leaf = np.arange(mid[-1] + 1, mid[-1] + 1 + 10_000)
        src += [np.full(100, h[-1]), np.repeat(mid, 100)]
        dst += [mid, leaf]
        n = int(leaf[-1]) + 1
        src.append([int(leaf[j])]); dst.append([n])
    n += 1
    ids = np.random.default_rng(6).permutation(n).astype(np.int32)
    e = graphgen.EdgeList(n, ids[np.concatenate(src)], ids[np.concatenate(dst)])
    ref = oracle.build_csr(e.n, e.src, e.dst)
    labels = oracle.components(ref)
    g = bfs.Graph.from_edges(e.src, e.dst, e.n)
    o = bfs.options(mode=bfs.MODE_TD_ONLY, cluster_size=cluster, timeout_ms=2000,
                    parent_mode=bfs.PARENT_MIN_ID if min_id else bfs.PARENT_ANY)
    roots = [int(ids[r]) for r in [start, n - 1] + tiny[:6]]
    want = {r: oracle.levels(ref, r) for r in roots}
    sched = {r: oracle.do_schedule(ref, want[r], oracle.MODE_TD) for r in roots}
    level, parent = _buffers(n)
    for r in roots:
        for _ in range(5):
            info = g.run(r, parent=parent, level=level, opts=o, stats=True, record_levels=64)
            pa = parent.cpu().numpy()
            assert np.array_equal(level.cpu().numpy(), want[r]), r
            assert oracle.certify(ref, r, want[r], pa, labels) == (0, -1), r
            assert not min_id or np.array_equal(pa, oracle.min_parent(ref, want[r])), r
            for col, name in enumerate(["dir", "nf", "mf", "nnext", "mnext"]):
                assert np.array_equal(info["records"][:, col], getattr(sched[r], name)), (r, name)
            clu = info["records"][:, 8] == -1
            assert clu.any() and (r in roots[2:] or not clu.all()), r
    outs = [torch.empty(n, dtype=torch.int32, device="cuda") for _ in range(200)]
    for i, out in enumerate(outs):
        g.run(int(ids[tiny[i % 60]]), level=out, opts=o)
    g.sync()
    for i, out in enumerate(outs):
        size = (2, 3, 21)[i % 60 % 3]
        lv = out.cpu().numpy()
        assert (lv >= 0).sum() == size and lv[ids[tiny[i % 60]]] == 0 and lv.max() == (1, 2, 1)[i % 60 % 3], i
    several = [int(ids[t]) for t in tiny[:30]]
    g.run_multiroot(several, parent=parent, level=level, opts=o)
    want = np.min(np.stack([np.where(x < 0, 1 << 30, x) for x in (oracle.levels(ref, r) for r in several)]), axis=0)
    assert np.array_equal(level.cpu().numpy(), np.where(want == 1 << 30, -1, want))
    g.close()


def test_multi_hub_behind_a_full_task_list(gpu_lib):
    """Bottom-up pulls of a batch where the rows of about 90 ids, one chunk task each, fill
    the task list before the longest row, the last id's, asks for its thousands: the answers,
    and that the row is not a chain of 16-id steps.  A step is one dependent read of ids and
    masks, 0.5 to 2 us: 2 M ids are 125,000 steps of 16 (over 62 ms a level) and 15,625 of
    128 (under 32 ms); the limit lies between."""
    import torch
    bfs = gpu_lib
    rows, leaves = 200_000, 2_000_000
    n = rows + leaves + 1
    r = graphgen.erdos_renyi(rows, 45 * rows, seed=9)
    leaf = np.arange(rows, rows + leaves, dtype=np.int32)
    e = graphgen.EdgeList(n, np.concatenate([r.src, np.full(leaves, n - 1, np.int32)]), np.concatenate([r.dst, leaf]))
    ref = oracle.build_csr(e.n, e.src, e.dst)
    deg = np.diff(ref.offsets)
    # rows longer than what a pull reads before it asks for a task, against the list's room
    assert (deg[:rows] > 72).sum() > ref.cols.size // 512 + ref.cols.size // 256 + 1024
    g = bfs.Graph.from_edges(e.src, e.dst, e.n)
    roots = [3, rows + 5, n - 1]
    level, parent = _buffers(n, len(roots))
    o = bfs.options(mode=bfs.MODE_BU_ONLY)
    g.run_multi(roots, level, parent=parent, opts=o)
    g.sync()
    want = [oracle.levels(ref, x) for x in roots]
    assert np.array_equal(level.cpu().numpy().reshape(-1, n), np.stack(want))
    assert np.array_equal(parent.cpu().numpy().reshape(-1, n), np.stack([oracle.min_parent(ref, w) for w in want]))
    # one search that never reaches the hub: every level scans its row to the end
    ev = [torch.cuda.Event(enable_timing=True) for _ in range(2)]
    took = []
    for _ in range(3):
        ev[0].record()
        g.run_multi(roots[:1], level[:n], opts=o)
        ev[1].record()
        ev[1].synchronize()
        took.append(ev[0].elapsed_time(ev[1]))
    levels = int(want[0].max()) + 1
    assert min(took) < 40.0 * levels, took
    g.close()


@pytest.mark.parametrize("k", [3, 64])
def test_multi_pull_lengths(gpu_lib, k):
    """Bottom-up pulls of rows of every length around where a group stops (72 ids), where it
    goes on to the end (136) and where one chunk task becomes two (584, 1096), starting on
    every offset of a 16-byte group."""
    bfs = gpu_lib
    rng = np.random.default_rng(k)
    lens = list(range(60, 150)) + [582, 583, 584, 585, 586, 648, 1095, 1096, 1097, 1160]
    m = 6000
    src = np.concatenate([np.full(d, i) for i, d in enumerate(lens)])
    dst = len(lens) + np.concatenate([rng.choice(m, d, replace=False) for d in lens])
    n = len(lens) + m
    ids = rng.permutation(n).astype(np.int32)
    e = graphgen.EdgeList(n, ids[src], ids[dst])
    ref = oracle.build_csr(e.n, e.src, e.dst)
    g = bfs.Graph.from_edges(e.src, e.dst, e.n, hub_first=True)
    roots = rng.choice(graphgen.pick_roots(e, 64, 5), k).tolist()
    want = np.stack([oracle.levels(ref, r) for r in roots])
    level, _ = _buffers(n, k)
    for mode in (bfs.MODE_BU_ONLY, bfs.MODE_DO):
        for rows in (bfs.BU_ROWS_BY_ID, bfs.BU_ROWS_HUB_FIRST):
            level.fill_(-7)
            g.run_multi(roots, level, opts=bfs.options(mode=mode, bu_rows=rows))
            g.sync()
            assert np.array_equal(level.cpu().numpy().reshape(k, n), want), (mode, rows)
    g.close()


@pytest.mark.parametrize("n", [31, 33, 155_649, 311_296, 622_597])
@pytest.mark.parametrize("k", [8, 9])
def test_multi_sizes_around_the_grid(gpu_lib, n, k):
    """Batches on graphs just below, above and at several times the grid's threads, with as
    many roots as write their rows as they go and one more (which keeps level planes)."""
    bfs = gpu_lib
    e = graphgen.erdos_renyi(n, 3 * n, seed=n)
    ref = oracle.build_csr(e.n, e.src, e.dst)
    g = bfs.Graph.from_edges(e.src, e.dst, e.n)
    roots = np.random.default_rng(n).choice(graphgen.pick_roots(e, 6, 5), k).tolist()
    lv = {r: oracle.levels(ref, r) for r in set(roots)}
    want = np.stack([lv[r] for r in roots])
    level, _ = _buffers(n, k)
    for mode in (bfs.MODE_DO, bfs.MODE_BU_ONLY, bfs.MODE_TD_ONLY):
        level.fill_(-7)
        g.run_multi(roots, level, opts=bfs.options(mode=mode))
        g.sync()
        assert np.array_equal(level.cpu().numpy().reshape(k, n), want), mode
    g.close()


@pytest.mark.parametrize("directed", [False, True])
@pytest.mark.parametrize("shape", ["er", "er_wide", "cap64", "cap65", "ladder", "path"])
def test_min_parents_of_short_rows(gpu_lib, shape, directed):
    """Minimum-id parents on graphs whose rows are short: levels that offer theirs edge by
    edge and levels that leave them to the pass after the last one, in one search; rows just
    within and past the length that allows it, and levels past the byte staging."""
    bfs = gpu_lib
    rng = np.random.default_rng(8)
    if shape.startswith("cap"):
        # a random graph and a star of 64 or 65 leaves among its vertices
        n, cap = 4000, int(shape[3:])
        e = graphgen.erdos_renyi(n, 3 * n, seed=8)
        keep = (e.src != 7) & (e.dst != 7)
        leaf = rng.choice(np.arange(8, n, dtype=np.int32), cap, replace=False)
        e = graphgen.EdgeList(n, np.concatenate([e.src[keep], np.full(cap, 7, np.int32)]),
                              np.concatenate([e.dst[keep], leaf]))
    else:
        e = {"er": lambda: graphgen.erdos_renyi(20_000, 160_000, seed=8),
             "er_wide": lambda: graphgen.erdos_renyi(300_001, 600_000, seed=8),
             "ladder": lambda: _mesh(3, 900, True, 3), "path": lambda: graphgen.path(600)}[shape]()
    if directed and shape in ("ladder", "path"):
        e = graphgen.EdgeList(e.n, np.concatenate([e.src, e.dst[::2]]), np.concatenate([e.dst, e.src[::2]]))
    if directed:
        out, inn = oracle.build_digraph(e.n, e.src, e.dst)
    else:
        out = inn = oracle.build_csr(e.n, e.src, e.dst)
    if shape.startswith("cap") and not directed:
        assert out.degree().max() == cap
    g = bfs.Graph.from_edges(e.src, e.dst, e.n, directed=directed)
    level, parent = _buffers(e.n)
    row = np.repeat(np.arange(e.n), np.diff(inn.offsets))
    for root in graphgen.pick_roots(e, 3, 2).tolist():
        _, want, _ = oracle.bfs_topdown(out, root)
        up = (want[row] > 0) & (want[inn.cols] == want[row] - 1)
        pmin = np.full(e.n, e.n, np.int64)
        np.minimum.at(pmin, row[up], inn.cols[up])
        pmin[pmin == e.n] = -1
        pmin[root] = root
        for mode in (bfs.MODE_TD_ONLY, bfs.MODE_DO, bfs.MODE_RANDOM):
            for with_level in (True, False):
                parent.fill_(-7)
                g.run(root, parent=parent, level=level if with_level else None,
                      opts=bfs.options(mode=mode, seed=5, parent_mode=bfs.PARENT_MIN_ID, cluster_size=1))
                g.sync()
                assert np.array_equal(parent.cpu().numpy(), pmin), (root, mode, with_level)
                assert not with_level or np.array_equal(level.cpu().numpy(), want), (root, mode)
    g.close()


@pytest.mark.parametrize("deg", [130, 140, 152, 300, 1100])
@pytest.mark.parametrize("long_rows", [1, 4, 5, 9, 0])
def test_bottom_up_long_rows_in_a_warp(gpu_lib, deg, long_rows):
    """Bottom-up searches with 1, 4, 5 and 9 rows past what the 4-lane groups read before the
    whole warp may take them, and with all rows (0) that long: levels, parents, counts."""
    bfs = gpu_lib
    rng = np.random.default_rng(deg + long_rows)
    n = 3000
    if long_rows == 0:
        e = graphgen.erdos_renyi(n, n * deg // 2, seed=deg)
    else:
        # the long rows' neighbours are the upper half; the search starts far from them
        h = np.arange(long_rows, dtype=np.int32)
        t = np.concatenate([rng.choice(np.arange(n // 2, n, dtype=np.int32), deg, replace=False) for _ in h])
        r = np.arange(long_rows, n, dtype=np.int32)
        ids = rng.permutation(n).astype(np.int32)
        e = graphgen.EdgeList(n, ids[np.concatenate([np.repeat(h, deg), r[:-1:7], r[:-3:5]])],
                              ids[np.concatenate([t, r[1::7], r[3::5]])])
    ref = oracle.build_csr(e.n, e.src, e.dst)
    labels = oracle.components(ref)
    g = bfs.Graph.from_edges(e.src, e.dst, e.n, hub_first=True)
    level, parent = _buffers(n)
    for root in graphgen.pick_roots(e, 2, 3).tolist() + [int(e.dst[0])]:
        want = oracle.levels(ref, root)
        for rows, scan in ((bfs.BU_ROWS_BY_ID, ref), (bfs.BU_ROWS_HUB_FIRST, oracle.hub_first(ref))):
            for mode, omode in ((bfs.MODE_BU_ONLY, oracle.MODE_BU), (bfs.MODE_DO, oracle.MODE_DO)):
                info = g.run(root, parent=parent, level=level, stats=True, record_levels=1024,
                             opts=bfs.options(mode=mode, bu_rows=rows))
                pa = parent.cpu().numpy()
                assert np.array_equal(level.cpu().numpy(), want), (root, mode, rows)
                assert oracle.certify(ref, root, want, pa, labels) == (0, -1), (root, mode, rows)
                s = oracle.do_schedule(scan, want, omode)
                for col, name in enumerate(["dir", "nf", "mf", "nnext", "mnext", "scanned", "examined"]):
                    assert np.array_equal(info["records"][:, col], getattr(s, name)), (root, mode, rows, name)
    g.close()


def test_multi_parents_at_the_planes_depth(gpu_lib):
    """A batch with parents whose deepest level is 13, 14 (the last one that the planes hold)
    and 15, on a graph with hubs: the answers, and that the one of 14 is served from the
    planes like the one of 13.  Past them the parents come from a scan of every row for
    every search, a hundred times the work here; one level more may double the planes' time."""
    import torch
    bfs = gpu_lib
    took = {}
    for depth in (13, 14, 15):
        r = graphgen.rmat(16, seed=1616)
        ref = oracle.build_csr(r.n, r.src, r.dst)
        hub = int(np.argmax(ref.degree()))
        far = oracle.levels(ref, hub)
        # a path on the hub: its end is `depth` levels from the vertices farthest from the hub
        tail = depth - int(far.max())
        assert tail > 0
        path = np.concatenate([[hub], np.arange(r.n, r.n + tail)]).astype(np.int32)
        e = graphgen.EdgeList(r.n + tail, np.concatenate([r.src, path[:-1]]), np.concatenate([r.dst, path[1:]]))
        ref = oracle.build_csr(e.n, e.src, e.dst)
        roots = [e.n - 1] * 2 + np.flatnonzero(far >= 0)[:30].tolist()
        want = np.stack([oracle.levels(ref, x) for x in roots])
        assert want.max() == depth
        g = bfs.Graph.from_edges(e.src, e.dst, e.n)
        level, parent = _buffers(e.n, len(roots))
        ev = [torch.cuda.Event(enable_timing=True) for _ in range(2)]
        for _ in range(4):
            ev[0].record()
            g.run_multi(roots, level, parent=parent)
            ev[1].record()
            ev[1].synchronize()
            took[depth] = min(took.get(depth, 1e9), ev[0].elapsed_time(ev[1]))
        assert np.array_equal(level.cpu().numpy().reshape(-1, e.n), want), depth
        assert np.array_equal(parent.cpu().numpy().reshape(-1, e.n),
                              np.stack([oracle.min_parent(ref, w) for w in want])), depth
        g.close()
    assert took[14] < 2 * took[13], took
