"""Weighted source kernel over the sizes at which its launch changes: 256, 512
and 1024 threads per block, and graphs too large for the settled bits in
shared memory; rows packed with their group, cut into chunks, and empty. BC
against the oracle within 1e-9 under the Eq. 4 pass and the vertex scan."""
import numpy as np
import pytest

import graphgen as gg
import oracle as O
from helpers import close, csr

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [97, 96 * 1024, 96 * 1024 + 1, 384 * 1024 + 1, 1_700_001])
def test_block_shapes(n):
    import paper_1708_08739_gb300 as bcd
    g = gg.erdos_renyi(n, 3 * n, 11)
    # a hub with a long row and many in-arcs, so that chunks and ties occur
    t, h = g.arcs()
    far = np.arange(1, min(n, 3000), dtype=np.int64)
    g = gg.csr_from_arcs(n, np.concatenate([t, np.zeros_like(far), far]), np.concatenate([h, far, np.zeros_like(far)]))
    g = g.with_weights(gg.uniform_weights(g.m, 1, 7, 12))
    og = O.Graph.from_csr(g)
    dg = bcd.bc_graph_create(g.n, g.offsets, g.cols, g.weights)
    specs = [{"r": 0, "kind": bcd.BC_QUERY_APPROX_T, "T": 12, "seed": 7},
             {"r": 5, "kind": bcd.BC_QUERY_APPROX_T, "T": 12, "seed": 7}]
    want = [O.bc_approx(og, s["r"], 12, 7)[0] for s in specs]
    for acc in (1, 3):
        for short in (1, 32):
            bcd.bc_set_config(dg, accumulation=acc, weighted_short_row=short, chunk_arcs=64)
            out, _ = bcd.bc_batch(dg, specs)
            for o, w in zip(out, want):
                assert o["status"] == 0 and close(o["bc"], w), (acc, short, o["bc"], w)
    dg.close()


@pytest.mark.parametrize("row", [0, 1, 31, 32, 33, 64, 128, 129, 1023, 1025])
def test_row_lengths(row):
    """One vertex with `row` out-arcs between a source fan and a sink, every
    arc tight, so each bit of the row's arc words counts."""
    import paper_1708_08739_gb300 as bcd
    arcs = [(0, 1), (1, 2)] + [(2, 4 + i) for i in range(row)] + [(4 + i, 3) for i in range(row)]
    n = 4 + max(row, 1)
    g = csr(n, arcs)
    g = g.with_weights(np.full(g.m, 3, dtype=np.uint32))
    og = O.Graph.from_csr(g)
    dg = bcd.bc_graph_create(g.n, g.offsets, g.cols, g.weights)
    for acc in (1, 2):
        bcd.bc_set_config(dg, accumulation=acc, chunk_arcs=32)
        for r in (1, 2):
            got, _ = bcd.bc_exact(dg, r)
            assert close(got, O.bc_exact(og, r, 0)[0]), (acc, r)
    dg.close()


@pytest.mark.parametrize("n,T,per_sm", [(5000, 64, 2), (32768, 64, 2), (32769, 64, 1), (100_000, 150, 1), (100_000, 400, 2),
                                        (400_000, 300, 1)])
def test_few_sources_on_wide_blocks(n, T, per_sm):
    """A launch of fewer sources than blocks takes wider blocks, fewer per SM;
    the empty slots of its last tile (up to 255) do not count as sources."""
    torch = pytest.importorskip("torch")
    import paper_1708_08739_gb300 as bcd
    g = gg.erdos_renyi(n, 3 * n, 11)
    g = g.with_weights(gg.uniform_weights(g.m, 1, 7, 12))
    og = O.Graph.from_csr(g)
    dg = bcd.bc_graph_create(g.n, g.offsets, g.cols, g.weights)
    r = int(gg.top_inout_vertices(g, 1)[0])
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    want = O.bc_approx(og, r, T, 7)[0]
    for acc in (2, 1):
        bcd.bc_set_config(dg, accumulation=acc)
        out, info = bcd.bc_batch(dg, [{"r": r, "kind": bcd.BC_QUERY_APPROX_T, "T": T, "seed": 7}])
        assert out[0]["status"] == 0 and close(out[0]["bc"], want), (acc, out)
        assert info["grid_blocks"] == per_sm * sms, (info["grid_blocks"], sms)
    dg.close()


@pytest.mark.parametrize("k", [1, 31, 33, 127, 129, 511, 512, 513, 1023, 1025, 4097])
def test_level_widths(k):
    """k vertices that settle at one distance, around the widths at which a
    block's warps draw further groups: three sources (wide blocks) and the k
    vertices themselves as sources."""
    import paper_1708_08739_gb300 as bcd
    arcs = [(0, 1), (1, 2), (2, 3)] + [(3, 5 + i) for i in range(k)] + [(5 + i, 4) for i in range(k)]
    arcs += [(4, 5 + k), (5 + k, 6 + k)]
    g = csr(7 + k, arcs)
    g = g.with_weights(np.full(g.m, 2, dtype=np.uint32))
    og = O.Graph.from_csr(g)
    dg = bcd.bc_graph_create(g.n, g.offsets, g.cols, g.weights)
    for acc in (1, 2):
        bcd.bc_set_config(dg, accumulation=acc)
        for r in (3, 4, 5 + k):
            got, _ = bcd.bc_exact(dg, r)
            assert close(got, O.bc_exact(og, r, 0)[0]), (acc, r)
    dg.close()
