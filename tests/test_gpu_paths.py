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
