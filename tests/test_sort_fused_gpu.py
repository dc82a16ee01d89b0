"""One-launch sorts (up to 524,288 keys) against numpy at the edges of the tiles
and of the launch's range, for every key and payload width, with digits that
all keys share (skipped passes), and inside a captured graph."""
import numpy as np
import pytest

from paper_2503_21937_gb300 import workloads as W

pytestmark = pytest.mark.gpu

SIZES = [2, 31, 33, 2047, 2048, 2049, 16385, 131072, 131073, 262144, 262145, 524288, 524289]


@pytest.fixture(scope="module")
def eng():
    import torch
    from paper_2503_21937_gb300 import Engine, build
    build.build()
    e = Engine()
    yield e
    e.close()
    torch.cuda.synchronize()


def _dev(a):
    import torch
    return torch.from_numpy(a.view(np.int32 if a.itemsize == 4 else np.int64).copy()).cuda()


@pytest.mark.parametrize("key,pay", [(4, 0), (4, 4), (4, 8), (8, 0), (8, 4), (8, 8)])
@pytest.mark.parametrize("n", SIZES)
def test_sizes_and_widths(eng, n, key, pay):
    s = W.stream(8000 + n % 91 + key + pay)
    kt, pt = (np.uint32, np.uint64)[key // 8], (np.uint32, np.uint64)[pay // 8]
    for bits in ((7, 17, 32) if key == 4 else (9, 40, 64)):
        raw = s.take(n)
        if bits < 64:
            raw &= np.uint64((1 << bits) - 1)
        if bits == 40:
            raw &= np.uint64(0xFF00FF0000)  # whole bytes that every key shares
        keys = raw.astype(kt)
        k = _dev(keys)
        order = np.argsort(keys, kind="stable")
        p = _dev(s.take(n).astype(pt)) if pay else None
        want = p.cpu().numpy().view(pt)[order] if pay else None
        eng.prim_sort(k, p, key_bits=bits)
        assert np.array_equal(k.cpu().numpy().view(kt), keys[order])
        if pay:
            assert np.array_equal(p.cpu().numpy().view(pt), want)


def test_noalloc_in_a_captured_graph():
    import torch
    from paper_2503_21937_gb300 import lobster
    s = W.stream(8100)
    rows = [np.stack([s.below(50000, 3000), s.below(50000, 40)]) for _ in range(3)]
    cols = _dev(rows[0])
    out, n_out = torch.zeros_like(cols), torch.zeros(1, dtype=torch.int64, device="cuda")
    assert lobster.unique_rows_noalloc(cols, out, n_out) == 0
    torch.cuda.synchronize()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g):
        assert lobster.unique_rows_noalloc(cols, out, n_out) == 0
    for r in rows:
        cols.copy_(_dev(r))
        g.replay()
        torch.cuda.synchronize()
        want = np.unique(r, axis=1)
        assert int(n_out.item()) == want.shape[1]
        assert np.array_equal(out[:, : want.shape[1]].cpu().numpy().view(np.uint32), want)


def test_each_noalloc_call_clears_its_barrier_words():
    """A call whose blocks wait on one another starts with a memset node (64 bytes of
    zeros) in the captured graph: it trusts nothing that an earlier call left.  (Calls
    that overlap, which could leave words behind, are not run.)"""
    import ctypes
    import torch
    from paper_2503_21937_gb300 import lobster
    cols = _dev(np.stack([W.stream(8200).below(50000, 3000)] * 2))
    out, n_out = torch.zeros_like(cols), torch.zeros(1, dtype=torch.int64, device="cuda")
    assert lobster.unique_rows_noalloc(cols, out, n_out) == 0
    torch.cuda.synchronize()
    if not hasattr(torch.cuda.CUDAGraph, "raw_cuda_graph"):
        pytest.skip("this torch does not give the captured graph")
    g = torch.cuda.CUDAGraph(keep_graph=True)
    with torch.cuda.graph(g):
        assert lobster.unique_rows_noalloc(cols, out, n_out) == 0
    cu = ctypes.CDLL("libcuda.so.1")
    h, n = ctypes.c_void_p(g.raw_cuda_graph()), ctypes.c_size_t(0)
    assert cu.cuGraphGetNodes(h, None, ctypes.byref(n)) == 0
    nodes = (ctypes.c_void_p * n.value)()
    assert cu.cuGraphGetNodes(h, nodes, ctypes.byref(n)) == 0
    kinds = []
    for node in nodes:
        t = ctypes.c_int(-1)
        assert cu.cuGraphNodeGetType(ctypes.c_void_p(node), ctypes.byref(t)) == 0
        kinds.append(t.value)
    assert sorted(kinds) == [0, 2], kinds  # one kernel, one memset
