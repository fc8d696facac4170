"""The one-launch pass of a small graph and the one-launch commit of a small
dense model, against the oracle and against the general kernels, at the edges
of their ranges.  Labels, counts and degrees are compared exactly, DL within
1e-12 (both sides sum x ln x exactly in fixed point at these sizes)."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

import oracle as O  # noqa: E402
import paper_2305_18663_gb300 as P  # noqa: E402
from synth.dcsbm import dcsbm, random_labels  # noqa: E402
from test_gpu_parity import _hub_graph, check_blockmodel, untraced_sweeps_vs_oracle  # noqa: E402

pytestmark = pytest.mark.gpu


def _same(a, b):
    assert np.array_equal(a.assignment(), b.assignment())
    ka, ca = a.coo()
    kb, cb = b.coo()
    assert np.array_equal(ka, kb) and np.array_equal(ca, cb)
    for x, y in zip(a.degrees(), b.degrees()):
        assert np.array_equal(x, y)
    assert a.dl() == b.dl()


# the last size that takes the one-launch pass and the first that does not
@pytest.mark.parametrize("n", [60_000, 60_001])
@pytest.mark.parametrize("dl_fp32", [0, 1])
def test_pass_at_its_line_equals_a_pass_in_parts(n, dl_fp32):
    # parts of the range never take it: their movers come from the lists
    g = dcsbm(n, 8 * n, 60, 2.5, 1, 100, 4.0, seed=1)
    b = random_labels(n, 60, seed=2)
    pg = P.Graph(g.n, g.src, g.dst)
    prm = P.Params.default(seed=4, dl_fp32=dl_fp32)
    whole, parts = P.Model(pg, 60, b, prm), P.Model(pg, 60, b, prm)
    for sw in range(3):
        st = whole.sweep(sw)
        for lo, hi in ((0, 1), (1, n // 3), (n // 3, n)):
            P.sbp_nodal_decide(parts.h, sw, lo, hi)
        sp = P.sbp_commit(parts.h)
        assert (st.n_proposed, st.n_moves, st.n_accepted, st.n_move_edges) == \
               (sp.n_proposed, sp.n_moves, sp.n_accepted, sp.n_move_edges)
        assert st.dl_after == sp.dl_after and st.dl_before == sp.dl_before
    _same(whole, parts)


# B around the one-launch commit's limit; few moves (update) and many (recount)
@pytest.mark.parametrize("B", [1, 2, 33, 512, 513])
@pytest.mark.parametrize("start", ["random", "near"])
def test_commit_equals_a_recount(B, start):
    g = dcsbm(3_000, 40_000, 12, 2.5, 1, 100, 4.0, seed=3)
    loops = np.arange(0, 300, dtype=np.int32)
    src, dst = np.concatenate([g.src, loops, g.src[:500]]), np.concatenate([g.dst, loops, g.dst[:500]])
    pg = P.Graph(g.n, src, dst)
    b = random_labels(g.n, B, seed=5) if start == "random" else (g.planted % B).astype(np.int32)
    one, full = P.Model(pg, B, b, P.Params.default(seed=6)), P.Model(pg, B, b, P.Params.default(seed=6, full_rebuild=1))
    om = O.Model(O.Graph(g.n, src, dst), B, b)
    for sw in range(5):
        a, c = one.sweep(sw), full.sweep(sw)
        assert a.as_dict() | {"n_recheck": 0} == c.as_dict() | {"n_recheck": 0}
        _same(one, full)
    om.set_b(B, one.assignment())
    check_blockmodel(one, om)
    # labels from outside: a nearby state, then one that moves most edges
    for frac in (0.01, 0.9):
        lab = one.assignment()
        pick = np.random.default_rng(7).random(g.n) < frac
        lab[pick] = random_labels(g.n, B, seed=8)[pick]
        P.sbp_set_assignment(one.h, B, lab)
        om.set_b(B, lab)
        check_blockmodel(one, om)


def test_hub_rows_of_a_small_graph():
    # rows of thousands of edges on one warp, several items per accepted hub
    g = _hub_graph()
    untraced_sweeps_vs_oracle(g, 40, random_labels(g.n, 40, seed=9), P.Graph(g.n, g.src, g.dst),
                              O.Graph(g.n, g.src, g.dst), "dense", sweeps=3)
