"""The allocation-free RV(r) kernel at the sizes where its split changes:
vertex counts around whole words and warps, rows around the length from which
a block walks them, long chains (many levels), and an empty reach set. Lists
bit-exact against the oracle."""
import ctypes as C

import numpy as np
import pytest

import graphgen as gg
import oracle as O
from helpers import csr

pytestmark = pytest.mark.gpu


def fan(n, row):
    """A chain 0 <- 1 <- 2 ... and a vertex with `row` in-arcs (from the last
    vertices) in its middle."""
    arcs = {(i + 1, i) for i in range(min(n - 1, 40))}
    hub = min(n - 1, 20)
    arcs |= {(n - 1 - i, hub) for i in range(min(row, n - 1)) if n - 1 - i != hub}
    return sorted(arcs)


@pytest.mark.parametrize("n,row", [(1, 0), (2, 0), (31, 3), (32, 3), (33, 3), (1100, 1023), (1100, 1024), (1100, 1025),
                                   (5000, 2049), (40000, 30000), (100001, 60000)])
def test_noalloc_edges(n, row):
    torch = pytest.importorskip("torch")
    import paper_1708_08739_gb300 as bcd
    g = csr(n, fan(n, row) if n > 1 else [])
    og = O.Graph.from_csr(g)
    roff, rcol = torch.from_numpy(og.roff.copy()).cuda(), torch.from_numpy(og.rcol.copy()).cuda()
    if rcol.numel() == 0:
        rcol = torch.zeros(1, dtype=torch.int32, device="cuda")
    out = torch.full((n + 1,), -7, dtype=torch.int32, device="cuda")
    for r in sorted({0, n - 1, n // 2, min(n - 1, 20)}):
        want = O.rv(og, r)
        k = bcd.bc_rv_compute_noalloc(roff.data_ptr(), rcol.data_ptr(), n, r, out.data_ptr(), n,
                                      torch.cuda.current_stream().cuda_stream)
        assert k == want.shape[0] and np.array_equal(out[:k].cpu().numpy(), want), (n, row, r)


def device_csr(og):
    torch = pytest.importorskip("torch")
    roff, rcol = torch.from_numpy(og.roff.copy()).cuda(), torch.from_numpy(og.rcol.copy()).cuda()
    return roff, rcol if rcol.numel() else torch.zeros(1, dtype=torch.int32, device="cuda")


@pytest.mark.parametrize("n,deg", [(300, 150), (2048, 127), (2048, 129), (4096, 500), (9001, 300)])
def test_noalloc_dense(n, deg):
    """Graphs whose arcs, not their vertices, decide how many blocks run."""
    torch = pytest.importorskip("torch")
    import paper_1708_08739_gb300 as bcd
    g = gg.erdos_renyi(n, n * deg, 5)
    og = O.Graph.from_csr(g)
    roff, rcol = device_csr(og)
    out = torch.full((n + 1,), -7, dtype=torch.int32, device="cuda")
    for r in (0, n // 3, n - 1):
        want = O.rv(og, r)
        k = bcd.bc_rv_compute_noalloc(roff.data_ptr(), rcol.data_ptr(), n, r, out.data_ptr(), n,
                                      torch.cuda.current_stream().cuda_stream)
        assert k == want.shape[0] and np.array_equal(out[:k].cpu().numpy(), want), (n, r)


@pytest.mark.parametrize("n,row", [(33, 3), (1100, 1025), (5000, 2049), (100001, 60000)])
def test_noalloc_writes_its_list_only(n, row):
    """Nothing past |RV| is written; a capacity of |RV| is enough, and with one
    less the call names the size and writes nothing."""
    torch = pytest.importorskip("torch")
    import paper_1708_08739_gb300 as bcd
    g = csr(n, fan(n, row))
    og = O.Graph.from_csr(g)
    roff, rcol = device_csr(og)
    stream = torch.cuda.current_stream().cuda_stream
    out = torch.empty(n + 64, dtype=torch.int32, device="cuda")
    for r in (0, n // 2, 20):
        want = O.rv(og, r)
        k = want.shape[0]
        for cap in sorted({k, n}):
            out.fill_(-7)
            got = bcd.bc_rv_compute_noalloc(roff.data_ptr(), rcol.data_ptr(), n, r, out.data_ptr(), cap, stream)
            host = out.cpu().numpy()
            assert got == k and np.array_equal(host[:k], want) and (host[k:] == -7).all(), (n, r, cap)
        if k > 0:
            out.fill_(-7)
            with pytest.raises(bcd.BCError) as e:
                bcd.bc_rv_compute_noalloc(roff.data_ptr(), rcol.data_ptr(), n, r, out.data_ptr(), k - 1, stream)
            assert e.value.status == bcd.BC_E_BUFFER_TOO_SMALL
            assert (out.cpu().numpy() == -7).all(), (n, r)
            cnt = C.c_int64(-1)
            st = bcd.lib().bc_rv_compute_noalloc(C.c_void_p(roff.data_ptr()), C.c_void_p(rcol.data_ptr()), n, r,
                                                 C.c_void_p(out.data_ptr()), k - 1, C.byref(cnt), C.c_void_p(stream))
            assert st == bcd.BC_E_BUFFER_TOO_SMALL and cnt.value == k, (n, r, cnt.value)
