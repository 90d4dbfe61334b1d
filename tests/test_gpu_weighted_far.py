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
