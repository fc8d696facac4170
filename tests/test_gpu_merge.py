"""The device's merge application and compaction against the oracle's.

The application is given the device's own proposals (checked elsewhere) and
has to make the same links as the oracle's sequential union, at the sizes
where its one-block and cluster forms meet and around their strides, for
scores that are all tied (a graph without edges: the order is the block id,
the links a random function with long cycles) and for scores that differ.
Everything compared is an integer.
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

import oracle as O  # noqa: E402
import paper_2305_18663_gb300 as P  # noqa: E402

pytestmark = pytest.mark.gpu


def _model(n, edges, seed, x):
    rng = np.random.default_rng(seed)
    src = rng.integers(0, n, edges).astype(np.int32)
    dst = rng.integers(0, n, edges).astype(np.int32)
    b = np.arange(n, dtype=np.int32)
    return P.Model(P.Graph(n, src, dst), n, b, P.Params.default(seed=seed, merge_proposals=x))


@pytest.mark.parametrize("degree", [0, 3])
@pytest.mark.parametrize("B", [2, 3, 33, 256, 1025, 4096, 4097, 20_011])
def test_application_equals_sequential_union(B, degree):
    for x in (1, 10):
        bs, bd = np.zeros(B, np.int32), np.zeros(B, np.float64)
        m = _model(B, degree * B, seed=B + x, x=x)
        P.sbp_merge_proposals(m.h, 5, bs, bd)
        most, _, _ = O.merge_apply(B, bs, bd, B)  # every link that closes no cycle
        for want in sorted({1, most // 2, most - 1, most} - {0, B}):
            P.sbp_set_assignment(m.h, B, np.arange(B, dtype=np.int32))
            done, mp, Bn = O.merge_apply(B, bs, bd, want)
            assert done == want
            got, rounds = P.sbp_merge_blocks(m.h, 5, want)
            assert (got, rounds) == (Bn, 1)
            assert np.array_equal(m.assignment(), mp)


@pytest.mark.parametrize("B", [5, 1024, 4097, 30_000])
def test_compaction_keeps_the_order(B):
    n = 2 * B
    rng = np.random.default_rng(B)
    b = rng.integers(0, B, n).astype(np.int32)  # about one block in seven is empty
    b[0] = B - 1
    m = P.Model(P.Graph(n, np.zeros(1, np.int32), np.ones(1, np.int32)), B, b)
    used, want = np.unique(b, return_inverse=True)
    assert P.sbp_compact(m.h) == used.size
    assert np.array_equal(m.assignment(), want)
