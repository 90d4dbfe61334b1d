"""The trial of the vertex scan (accumulation 4, a hub among the query
vertices): the terms of a group's first tile are counted before any is added,
and above 2^23 of them, and a sixteenth of the tight pairs, every tile is left
to Eq. 4. A hub with arcs from and to every spoke has about (sources of the
tile) x (spokes) terms, since the shortest paths between spokes run through it;
a long chain into the hub and one out of it put query vertices at levels past
63, where the count keeps one class. Scores within 1e-9 of the oracle on every
route."""
import time

import pytest

import oracle as O
from helpers import close, csr

pytestmark = pytest.mark.gpu


def hub(spokes, into, out):
    """(n, arcs, first vertex of the chain out of the hub): hub 0, spokes 1 ..
    spokes, a chain of `into` vertices into the hub, one of `out` out of it."""
    arcs = [(0, i) for i in range(1, spokes + 1)] + [(i, 0) for i in range(1, spokes + 1)]
    arcs += [(i, i + 1) for i in range(1, spokes)]
    a, c = spokes + 1, spokes + 1 + into
    arcs += [(a + i, a + i + 1) for i in range(into - 1)] + [(a + into - 1, 0)]
    arcs += [(0, c)] + [(c + i, c + i + 1) for i in range(out - 1)]
    return c + out, arcs, c


# The terms of the first tile: (its sources that the hub's query needs) x (spokes) or a little more. Spokes, chain in,
# chain out, draws of the queries at the hub and a spoke, draws of the one behind it, tiles, scan left to Eq. 4 (the
# first: 100 x 60,000 is below 2^23, the second 200 x 60,000 above).
CASES = [(60000, 5, 200, 100, 100, 1, False), (60000, 5, 200, 200, 8, 1, True), (60000, 5, 200, 600, 8, 3, True),
         (40000, 2000, 200, 240, 8, 1, True), (40000, 2000, 200, 700, 8, 3, True), (3000, 700, 200, 100, 8, 1, False),
         (3000, 700, 200, 400, 8, 2, False)]


@pytest.mark.parametrize("spokes,into,out,T,Tc,tiles,left", CASES)
def test_trial(spokes, into, out, T, Tc, tiles, left):
    import paper_1708_08739_gb300 as bcd
    n, arcs, c = hub(spokes, into, out)
    g = csr(n, arcs)
    og = O.Graph.from_csr(g)
    dg = bcd.bc_graph_create(g.n, g.offsets, g.cols)
    rs = [0, 17, c + 150]
    specs = [{"r": r, "kind": bcd.BC_QUERY_APPROX_T, "T": t, "seed": 7} for r, t in zip(rs, (T, T, Tc))]
    want = [O.bc_approx(og, s["r"], s["T"], 7, 0)[0] for s in specs]

    def check(out):
        for r, o, w in zip(rs, out, want):
            assert o["status"] == 0 and o["flags"] == 0 and close(o["bc"], w), (r, o, w)

    for _ in range(2):  # the second call starts from what the first left behind
        res, info = bcd.bc_batch(dg, specs)
        check(res)
        assert info["tiles"] == tiles, info
        assert (info["scan_tiles"] == 0) == left, info
    # without the hub the same handle scans, and then tries again
    res, info = bcd.bc_batch(dg, specs[1:])
    assert info["scan_tiles"] == info["tiles"], info
    for o, w in zip(res, want[1:]):
        assert close(o["bc"], w)
    check(bcd.bc_batch(dg, specs)[0])
    # two shards of the group
    parts = [bcd.bc_batch_shard(dg, specs, k, 2)[0] for k in range(2)]
    for i, w in enumerate(want):
        assert close(sum(p[i]["bc"] for p in parts), w), (i, w)
    # the serving loop's slices
    srv = bcd.Server(dg, tiles_per_slice=2)
    for _ in range(2):
        tickets = [srv.submit(s) for s in specs]
        got, deadline = [None] * len(specs), time.time() + 120
        while any(x is None for x in got) and time.time() < deadline:
            for i, t in enumerate(tickets):
                if got[i] is None:
                    x = srv.poll(t, timeout_us=100000)
                    got[i] = None if x is None else x[0]
        assert all(x is not None for x in got)
        check(got)
    srv.close()
    dg.close()
