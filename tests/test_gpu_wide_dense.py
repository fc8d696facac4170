"""The prefix rows of a dense model at many blocks against the oracle, around
the size they take over at and the tiles they are made in: counts, degrees and
DL directly, prefixes and pivots through the proposals that search them.
Integers are compared exactly, DL within 1e-12."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

import oracle as O  # noqa: E402
import paper_2305_18663_gb300 as P  # noqa: E402
from synth.dcsbm import dcsbm  # noqa: E402
from test_gpu_parity import check_blockmodel, run_sweeps  # noqa: E402

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("B", [1025, 1399, 1400, 1401, 2304, 3001])
def test_wide_prefix_matches_oracle(B):
    g = dcsbm(4000, 60_000, 20, 2.1, 1, 400, 3.0, seed=B)
    b = (np.random.default_rng(B).random(g.n) ** 3 * B).astype(np.int32)  # crowded and empty blocks
    pm, om, _ = run_sweeps(g, B, b, sweeps=2)
    bs, bd = np.zeros(B, np.int32), np.zeros(B, np.float64)
    P.sbp_merge_proposals(pm.h, 3, bs, bd)
    obs, obd = om.merge_proposals(7, 3, 10)
    assert np.all(np.abs(bd - obd) <= 1e-9 * np.maximum(np.abs(obd), 1.0))
    assert (bs != obs).sum() <= max(2, B // 200)  # ties on the score grid
    om.set_b(B, pm.assignment())
    check_blockmodel(pm, om)


def test_growing_a_dense_model_past_the_line():
    g = dcsbm(3000, 30_000, 10, 2.5, 1, 100, 4.0, seed=1)
    pg, G = P.Graph(g.n, g.src, g.dst), O.Graph(g.n, g.src, g.dst)
    m = P.Model(pg, 500, (np.arange(g.n) % 500).astype(np.int32))
    for B in (1500, 700, 2500, 1400):
        b = (np.arange(g.n) * 7 % B).astype(np.int32)
        P.sbp_set_assignment(m.h, B, b)
        check_blockmodel(m, O.Model(G, B, b))


@pytest.mark.parametrize("B", [1599, 1600, 1601])
def test_both_sides_of_the_line(B):
    test_wide_prefix_matches_oracle(B)
    # and the column sums of a model that grows past it
    g = dcsbm(3000, 30_000, 10, 2.5, 1, 100, 4.0, seed=2)
    m = P.Model(P.Graph(g.n, g.src, g.dst), 700, (np.arange(g.n) % 700).astype(np.int32))
    b = (np.arange(g.n) * 7 % B).astype(np.int32)
    P.sbp_set_assignment(m.h, B, b)
    check_blockmodel(m, O.Model(O.Graph(g.n, g.src, g.dst), B, b))
