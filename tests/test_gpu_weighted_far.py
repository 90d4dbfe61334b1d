"""Weighted distances around and past 2^24 - 1, the largest that the source
kernel's narrow layout holds (its code for an unreached vertex is 2^24 - 1):
the launch has to rerun on 16-byte pairs whether an offer hits that value or
steps over it. Directed paths, where BC(r) = r (n - 1 - r) whatever the
weights; the scores are integers that every path sums exactly up to rounding
(1e-9)."""
import numpy as np
import pytest

from helpers import close

pytestmark = pytest.mark.gpu


def path_graph(weights):
    import paper_1708_08739_gb300 as bcd
    n = len(weights) + 1
    off = np.append(np.arange(n), n - 1).astype(np.int64)
    return n, bcd.bc_graph_create(n, off, np.arange(1, n, dtype=np.int32), np.asarray(weights, dtype=np.uint32))


def check(dg, n, vertices):
    import paper_1708_08739_gb300 as bcd
    for acc in (4, 2, 3, 1):
        bcd.bc_set_config(dg, accumulation=acc)
        out, _ = bcd.bc_batch(dg, [{"r": r} for r in vertices])
        for r, o in zip(vertices, out):
            assert o["status"] == 0 and close(o["bc"], r * (n - 1 - r)), (acc, r, o["bc"])
        r = vertices[-1]
        assert close(bcd.bc_exact(dg, r)[0], r * (n - 1 - r)), (acc, r)


@pytest.mark.parametrize("past", [-2, -1, 0, 1, 1900])
def test_distance_limit(past):
    """The path's length is 2^24 + past: 4,096 arcs of 4,095, one of 2,000
    and the rest."""
    n, dg = path_graph([4095] * 4096 + [2000, (1 << 24) + past - 4096 * 4095 - 2000])
    check(dg, n, [3, n - 2])
    dg.close()


@pytest.mark.parametrize("weight", [4000, 4095])
def test_long_paths(weight):
    n, dg = path_graph([weight] * 9999)
    check(dg, n, [9000, 5000])
    dg.close()


@pytest.mark.parametrize("top", [2, 255, 4095])
@pytest.mark.parametrize("threads", [128, 512])
@pytest.mark.parametrize("kernel", [1, 2])
def test_far_apart_distances(kernel, threads, top):
    """Few pending vertices with distances up to the largest weight apart, so
    that a level's offers land in ring slots of smaller distances: every block of
    the tile kernel (with kernel 2 it runs the query vertices' own traversal) has
    to find the same next distance, whichever is ahead."""
    import graphgen as gg
    import oracle as O
    import paper_1708_08739_gb300 as bcd
    rng = np.random.default_rng(top)
    n, dg = path_graph(rng.integers(max(1, top // 2), top + 1, 250))
    for acc in (4, 1):
        bcd.bc_set_config(dg, accumulation=acc, weighted_kernel=kernel, block_threads=threads, weighted_words=1)
        out, _ = bcd.bc_batch(dg, [{"r": r} for r in (30, 230)])
        for r, o in zip((30, 230), out):
            assert o["status"] == 0 and close(o["bc"], r * (n - 1 - r)), (acc, r, o)
        assert close(bcd.bc_exact(dg, 60)[0], 60 * (n - 61)), acc
    dg.close()
    g = gg.erdos_renyi(500, 700, 4)
    g = g.with_weights(gg.uniform_weights(g.m, max(1, top // 2), top, 3))
    og = O.Graph.from_csr(g)
    dg = bcd.bc_graph_create(g.n, g.offsets, g.cols, g.weights)
    rs = [int(x) for x in gg.top_inout_vertices(g, 2)]
    for acc in (4, 1):
        bcd.bc_set_config(dg, accumulation=acc, weighted_kernel=kernel, block_threads=threads)
        out, _ = bcd.bc_batch(dg, [{"r": r} for r in rs])
        for r, o in zip(rs, out):
            assert o["status"] == 0 and close(o["bc"], O.bc_exact(og, r, 0)[0]), (acc, r)
    dg.close()
