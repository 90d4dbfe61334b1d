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
