"""The sparse rows at more than 1024 blocks against the oracle: every kernel
of the row build at the edges of its range (rows of 0, 1, 32, 33, 64, 65,
128, 129, 512, 513, 4096, 4097, 16,384 and 16,385 labels and more; many repeats and none; windows of
columns), as counts, degrees and DL, and through the proposals and lookups
that read the rows (sweeps and a merge round)."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

import oracle as O  # noqa: E402
import paper_2305_18663_gb300 as P  # noqa: E402
from test_gpu_parity import _G, check_blockmodel, untraced_sweeps_vs_oracle  # noqa: E402

pytestmark = pytest.mark.gpu

SIZES = (0, 1, 2, 31, 32, 33, 63, 64, 65, 127, 128, 129, 255, 256, 257, 511, 512, 513, 1000, 4095, 4096, 4097, 9000, 16_384, 16_385, 40_000)


def _graph(n, spread, seed):
    """vertices 0..: an out-row of every size, then an in-row of every size;
    `spread`: far ends over all vertices, else over a few (repeats)"""
    rng = np.random.default_rng(seed)
    src, dst = [np.arange(n - 1)], [np.arange(1, n)]  # no block without edges but those of size 0
    for i, k in enumerate(SIZES):
        far = rng.integers(0, n if spread else 40, k)
        src += [np.full(k, 100 + i), far]
        dst += [far, np.full(k, 200 + i)]
    return _G(n, np.concatenate(src), np.concatenate(dst))


@pytest.mark.parametrize("spread", [False, True])
@pytest.mark.parametrize("n,B", [(1500, 1025), (5000, 5000), (9000, 8192), (9000, 8193), (40_000, 40_000), (40_000, 33_000)])
def test_rows_match_oracle(n, B, spread):
    g = _graph(n, spread, seed=n + B)
    b = (np.arange(n) % B).astype(np.int32)
    m = P.Model(P.Graph(g.n, g.src, g.dst), B, b, P.Params.default(seed=1, dense_max_B=1))
    om = O.Model(O.Graph(g.n, g.src, g.dst), B, b)
    check_blockmodel(m, om)
    # and again over what the first build left, from other labels
    b = ((np.arange(n) * 7 + 3) % B).astype(np.int32)
    P.sbp_set_assignment(m.h, B, b)
    om.set_b(B, b)
    check_blockmodel(m, om)


@pytest.mark.parametrize("n,B", [(1500, 1025), (5000, 4500)])
def test_sweeps_and_merges_on_the_rows(n, B):
    g = _graph(n, True, seed=n)
    b = np.random.default_rng(2).integers(0, B, n).astype(np.int32)  # some blocks are empty
    b[: n // 20] = 5
    pg, G = P.Graph(g.n, g.src, g.dst), O.Graph(g.n, g.src, g.dst)
    untraced_sweeps_vs_oracle(g, B, b, pg, G, "sparse", sweeps=3, seed=3)
    m = P.Model(pg, B, b, P.Params.default(seed=4, dense_max_B=1))
    om = O.Model(G, B, b)
    oB, orounds = om.merge_phase(O.Params(seed=4), 7, B // 3)
    assert P.sbp_merge_blocks(m.h, 7, B // 3) == (oB, orounds)
    assert np.array_equal(m.assignment(), om.assignment())
    check_blockmodel(m, om)


@pytest.mark.parametrize("n,B", [(1500, 1025), (40_000, 33_000)])
def test_reading_the_nonzeros_leaves_the_rows_as_they_are(n, B):
    # many edges a nonzero (repeats), so most slots of the rows are empty; the
    # packing uses scratch of the build
    g = _graph(n, False, seed=n)
    pg, om = P.Graph(g.n, g.src, g.dst), O.Model(O.Graph(g.n, g.src, g.dst), B, (np.arange(n) % B).astype(np.int32))
    read, not_read = (P.Model(pg, B, om.assignment(), P.Params.default(seed=1, dense_max_B=1)) for _ in range(2))
    launches = P.sbp_kernel_launches()
    keys, cnt = read.coo()
    assert P.sbp_kernel_launches() > launches  # packed on the device, not read with the slack
    okeys, ocnt = om.coo()
    assert np.array_equal(keys, okeys) and np.array_equal(cnt, ocnt)
    for sw in range(2):
        a, c = read.sweep(sw), not_read.sweep(sw)
        assert a.as_dict() == c.as_dict()
        read.coo()
    om.set_b(B, read.assignment())
    check_blockmodel(read, om)
    check_blockmodel(not_read, om)
