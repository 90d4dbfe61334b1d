"""A handle's first call that overflows several things in one launch: the
level history, which starts at 8 n + 4,096 entries and doubles (a 256-source
tile on a path needs 256 n, five doublings), and the 32-bit path counts, which
a chain of 26 diamonds (sigma 2^26) takes past their limit. Scores within 1e-9
of the oracle on the first call, not only on a second one."""
import numpy as np
import pytest

import oracle as O
from helpers import close, csr

pytestmark = pytest.mark.gpu


def path_and_diamonds(length, k):
    """(n, arcs, r): a path of `length` vertices, k diamonds, r, a vertex."""
    arcs, at, n = [(i, i + 1) for i in range(length - 1)], length - 1, length
    for _ in range(k):
        b, c, d = n, n + 1, n + 2
        n += 3
        arcs += [(at, b), (at, c), (b, d), (c, d)]
        at = d
    return n + 2, arcs + [(at, n), (n, n + 1)], n


@pytest.mark.parametrize("acc", [4, 1])
@pytest.mark.parametrize("diamonds", [20, 25, 26, 27])
def test_history_and_counts_on_a_first_call(diamonds, acc):
    import paper_1708_08739_gb300 as bcd
    n, arcs, r = path_and_diamonds(2000, diamonds)
    g = csr(n, arcs)
    og = O.Graph.from_csr(g)
    dg = bcd.bc_graph_create(g.n, g.offsets, g.cols)
    bcd.bc_set_config(dg, accumulation=acc)
    want = O.bc_exact(og, r, 0)[0]
    for _ in range(2):
        got, info = bcd.bc_exact(dg, r)
        assert close(got, want) and info["flags"] == 0, (got, want)
    dg.close()


@pytest.mark.parametrize("words,threads", [(1, 128), (4, 256), (16, 256), (16, 512)])
@pytest.mark.parametrize("kernel", [1, 2])
def test_weighted_lists_overflow_on_a_first_call(kernel, words, threads):
    """Dense layers and rows that are all cut: in the tile kernel one level
    overflows the chunk list and the next the ring slot. Every block has to
    leave at the barrier behind an overflow, whichever block met it."""
    import paper_1708_08739_gb300 as bcd
    width, depth = 59, 9
    rng = np.random.default_rng(3)
    arcs = [(width * k + i, width * (k + 1) + j) for k in range(depth - 1) for i in range(width) for j in range(width)
            if rng.random() < 0.6]
    arcs += [(width * (depth - 1) + i, i) for i in range(width)]
    g = csr(width * depth, arcs)
    g = g.with_weights(rng.integers(1, 3, g.m).astype(np.uint32))
    og = O.Graph.from_csr(g)
    r = 229
    want = O.bc_exact(og, r, 0)[0]
    for acc in (1, 4):
        dg = bcd.bc_graph_create(g.n, g.offsets, g.cols, g.weights)
        bcd.bc_set_config(dg, accumulation=acc, weighted_kernel=kernel, weighted_words=words, block_threads=threads,
                          weighted_short_row=8)
        assert close(bcd.bc_exact(dg, r)[0], want), acc
        out, _ = bcd.bc_batch(dg, [{"r": r}, {"r": 10}])
        assert close(out[0]["bc"], want) and close(out[1]["bc"], O.bc_exact(og, 10, 0)[0]), acc
        dg.close()


@pytest.mark.parametrize("words,threads", [(1, 128), (2, 256), (4, 512), (8, 512)])
def test_lists_overflow_again_and_again(words, threads):
    """The same for the unweighted kernel: a lattice, whose sources meet the
    vertices at many levels, with counts past 2^26 and several teams."""
    import paper_1708_08739_gb300 as bcd
    a, b = 20, 36  # corner to corner C(54, 19), below 2^53
    arcs = [(i * b + j, i * b + j + 1) for i in range(a) for j in range(b - 1)]
    arcs += [(i * b + j, (i + 1) * b + j) for i in range(a - 1) for j in range(b)]
    g = csr(a * b, arcs + [(y, x) for x, y in arcs])
    og = O.Graph.from_csr(g)
    r = 10 * b + 12
    w300 = O.bc_approx(og, r, 300, 7, 0)
    for acc in (4, 1):
        dg = bcd.bc_graph_create(g.n, g.offsets, g.cols)
        bcd.bc_set_config(dg, accumulation=acc, tile_words=words, block_threads=threads, chunk_arcs=32)
        got, info = bcd.bc_approx_T(dg, r, 300, 7)
        assert info["flags"] == 0 and w300[3] == 0 and close(got, w300[0]), acc
        dg.close()
