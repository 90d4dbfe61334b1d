"""Path counts at the edge of their 32-bit form (unweighted graphs).

The forward pass holds sigma as 32-bit integers trusted below 2^26 and reruns
in fp64 when a count reaches that. A chain of k diamonds doubles sigma k
times; behind it a fan of 40 in-arcs (more than one 32-arc chunk) and one of
31 (a whole chunk less one) multiply it, so that single rows, partial sums and
their total cross the limit for different k. Integers below 2^53: bit-exact
against the oracle on both sides of the limit, and dependencies within 1e-9
(ratios and sums of fp64 numbers in another order).
"""
import numpy as np
import pytest

import oracle as O
from helpers import close, csr

pytestmark = pytest.mark.gpu


def diamonds(k):
    """(n, arcs, a query vertex in the chain, the last vertex): k diamonds,
    a fan of 40 into one vertex, a fan of 31 into the next, and a tail."""
    arcs, at, n = [], 0, 1
    for _ in range(k):
        b, c, d = n, n + 1, n + 2
        n += 3
        arcs += [(at, b), (at, c), (b, d), (c, d)]
        at = d
    mid = at
    for width in (40, 31):
        y = n + width
        for i in range(width):
            arcs += [(at, n + i), (n + i, y)]
        n = y + 1
        at = y
    arcs += [(at, n), (n, n + 1)]
    return n + 2, arcs, mid, at


@pytest.mark.parametrize("words,chunk", [(1, 32), (2, 32), (4, 32), (8, 32), (4, 128), (2, 64)])
@pytest.mark.parametrize("k", [19, 20, 21, 25, 26, 27, 35])
def test_counts_around_the_limit(words, chunk, k):
    import paper_1708_08739_gb300 as bcd
    n, arcs, mid, last = diamonds(k)
    g = csr(n, arcs)
    og = O.Graph.from_csr(g)
    dg = bcd.bc_graph_create(g.n, g.offsets, g.cols)
    bcd.bc_set_config(dg, tile_words=words, chunk_arcs=chunk, accumulation=1)
    srcs = np.array([0, 1, 3, 6, mid], dtype=np.int32)
    tgts = np.array([mid, last, 3], dtype=np.int32)
    odep, _, _ = O.dependencies(og, srcs, tgts, 0)
    for _ in range(2):  # the second call starts in the form the first ended in
        dist, sig, dep, flags = bcd.bc_spd_probe(dg, srcs, tgts)
        for i, s in enumerate(srcs.tolist()):
            st = O.source_state(og, s)
            assert np.array_equal(dist[i], st["dist"]), s
            assert np.array_equal(sig[i], st["sigma"]), s
            assert flags[i] == 0
            for j, t in enumerate(tgts.tolist()):
                if t != s:
                    assert close(dep[i, j], odep[i, j]), (s, t)
    for acc in (1, 2, 3):
        bcd.bc_set_config(dg, accumulation=acc)
        out, _ = bcd.bc_batch(dg, [{"r": mid}, {"r": last}])
        for r, o in zip((mid, last), out):
            assert o["status"] == 0 and close(o["bc"], O.bc_exact(og, r, 0)[0]), (acc, r)
        got, _ = bcd.bc_exact(dg, mid)
        assert close(got, O.bc_exact(og, mid, 0)[0]), acc
    dg.close()


def test_chunk_size_and_width_changes_between_calls():
    """Rows that one chunk size sums in registers and another in atomic adds,
    and slabs of another width, on one handle: sigma exact after each change."""
    import graphgen as gg
    import paper_1708_08739_gb300 as bcd
    g = gg.rmat(10, 12, seed=4)
    og = O.Graph.from_csr(g)
    dg = bcd.bc_graph_create(g.n, g.offsets, g.cols)
    srcs = np.flatnonzero(g.out_degree() > 0)[:70].astype(np.int32)
    want = [O.source_state(og, int(s)) for s in srcs[:48]]
    top = int(gg.top_inout_vertices(g, 1)[0])
    bc = O.bc_exact(og, top, 0)[0]
    for words, chunk in [(4, 256), (4, 32), (2, 32), (2, 128), (8, 32), (1, 64), (4, 32)]:
        bcd.bc_set_config(dg, tile_words=words, chunk_arcs=chunk)
        assert close(bcd.bc_exact(dg, top)[0], bc), (words, chunk)
        dist, sig, _, _ = bcd.bc_spd_probe(dg, srcs[:48], [], want_dep=False)
        for i, st in enumerate(want):
            assert np.array_equal(dist[i], st["dist"]) and np.array_equal(sig[i], st["sigma"]), (words, chunk, i)
    dg.close()
