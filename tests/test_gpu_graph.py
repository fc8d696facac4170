"""The device build of the graph (sbp_load_graph) against the oracle's rows.

The rows are read through what depends on them: a traced sweep picks the
j-th edge end of every vertex (row order, duplicates and self-loops kept),
the commits after it follow the twins of the moved vertices' edges, the
kernels of the degree groups walk the group order, and a hybrid pass visits
vertices by descending degree with ties by id.  Integers are compared
exactly, Delta DL as in test_gpu_parity.
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

import oracle as O  # noqa: E402
import paper_2305_18663_gb300 as P  # noqa: E402
from test_gpu_parity import check_blockmodel, run_sweeps  # noqa: E402

pytestmark = pytest.mark.gpu


class _G:
    def __init__(self, n, src, dst):
        self.n, self.src, self.dst = n, np.ascontiguousarray(src, np.int32), np.ascontiguousarray(dst, np.int32)


def _multigraph(n, m, seed):
    """edges with repeats, self-loops, isolated vertices and, for the larger
    graphs, rows of every degree group"""
    rng = np.random.default_rng(seed)
    live = max(1, n // 2)
    src, dst = rng.integers(0, live, m), rng.integers(0, live, m)
    hubs = rng.integers(0, min(live, 4), m // 4)
    src[: m // 4] = hubs
    dst[m // 4: m // 2] = np.where(rng.random(m // 2 - m // 4) < 0.1, src[m // 4: m // 2], dst[m // 4: m // 2])
    src[-m // 8:], dst[-m // 8:] = src[: m // 8 + (m % 8 > 0)], dst[: m // 8 + (m % 8 > 0)]  # repeats
    return _G(n, src, dst)


# n * n on both sides of 2^32 (32- and 64-bit edge keys); one edge; edges of
# several sort chunks
@pytest.mark.parametrize("n,m", [(1, 3), (2, 1), (300, 4097), (65_536, 20_000), (65_537, 20_000), (5_000, 300_001)])
def test_rows_of_a_multigraph(n, m):
    g = _multigraph(n, m, seed=n + m)
    B = min(n, 7)
    b = np.random.default_rng(n).integers(0, B, n).astype(np.int32)
    run_sweeps(g, B, b, sweeps=2)


def test_device_and_host_edges_give_the_same_graph():
    g = _multigraph(3_000, 40_000, seed=5)
    b = (np.arange(g.n) % 11).astype(np.int32)
    prm = P.Params.default(seed=3, hybrid_h=500)  # visits by_degree
    models = []
    for s, d in ((g.src, g.dst), (torch.from_numpy(g.src).cuda(), torch.from_numpy(g.dst).cuda()),
                 (g.src, torch.from_numpy(g.dst).cuda())):
        m = P.Model(P.Graph(g.n, s, d), 11, b, prm)
        for i in range(3):
            m.sweep(i)
        models.append(m)
    om = O.Model(O.Graph(g.n, g.src, g.dst), 11, models[0].assignment())
    for m in models:
        assert np.array_equal(m.assignment(), models[0].assignment())
        check_blockmodel(m, om)


@pytest.mark.parametrize("device", [False, True])
def test_first_bad_edge_is_named(device):
    src = np.array([0, 1, 2, 5, -1], np.int32)
    dst = np.array([1, 2, 0, 0, 0], np.int32)
    if device:
        src, dst = torch.from_numpy(src).cuda(), torch.from_numpy(dst).cuda()
    with pytest.raises(P.SbpError, match="at edge 3"):
        P.Graph(5, src, dst)


def _pool_high(call):
    """bytes that `call` took from the device's memory pool at the most"""
    import ctypes
    import os

    for lib in ("libcudart.so.13", "libcudart.so", "/usr/local/cuda/lib64/libcudart.so"):
        try:
            rt = ctypes.CDLL(lib)
            break
        except OSError:
            continue
    else:
        pytest.skip("no CUDA runtime library to ask")
    pool, zero, high, now = ctypes.c_void_p(), ctypes.c_uint64(0), ctypes.c_uint64(0), ctypes.c_uint64(0)
    dev = torch.cuda.current_device()
    assert rt.cudaDeviceGetDefaultMemPool(ctypes.byref(pool), dev) == 0
    torch.cuda.synchronize()
    assert rt.cudaMemPoolSetAttribute(pool, 8, ctypes.byref(zero)) == 0  # cudaMemPoolAttrUsedMemHigh
    assert rt.cudaMemPoolGetAttribute(pool, 7, ctypes.byref(now)) == 0  # cudaMemPoolAttrUsedMemCurrent
    call()
    torch.cuda.synchronize()
    assert rt.cudaMemPoolGetAttribute(pool, 8, ctypes.byref(high)) == 0
    return high.value - now.value


@pytest.mark.parametrize("device", [False, True])
@pytest.mark.parametrize("n,m", [(1_000, 3_000_000), (70_000, 3_000_000), (1_000_000, 100_000)])
def test_loading_holds_no_scratch_of_the_edges_size(n, m, device):
    g = _multigraph(n, m, seed=n)
    src, dst = (torch.from_numpy(x).cuda() if device else x for x in (g.src, g.dst))
    assert 16 * n < _pool_high(lambda: P.Graph(n, src, dst)) <= 16 * n + (5 << 20)
