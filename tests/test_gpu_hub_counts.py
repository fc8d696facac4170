"""A vertex with 32,768 to 65,535 in-edges from one block: its counts towards
its own block r and the proposed block s are held as 16-bit halves of one
word, and both halves are unsigned.  Hubs that have such a count towards r and
hubs that have it towards s decide as the oracle does, in the one-launch pass,
in the degree groups' kernels and in the batched searches."""
import os

import numpy as np
import pytest

torch = pytest.importorskip("torch")

import oracle as O  # noqa: E402
import paper_2305_18663_gb300 as P  # noqa: E402
from test_gpu_parity import TOL, _G, check_blockmodel  # noqa: E402

pytestmark = pytest.mark.gpu
NT = max(1, min(16, os.cpu_count() or 1))
HUB_EDGES = 40_000


def hub_graph(n, seed=0):
    """(graph, planted labels, labels to start from): edges from block 0 into
    block 1 and from there into the loose block 3, edges inside block 2.  Two hubs of block 1 start
    in block 0, where all their in-edges come from (40,000 towards r); two hubs
    of block 2 start in block 3 (40,000 in-edges towards s)."""
    rng = np.random.default_rng(seed)
    planted = (np.arange(n) % 4).astype(np.int32)
    of = [np.flatnonzero(planted == q) for q in range(4)]
    hubs_r, hubs_s = of[1][:2], of[2][:2]
    src = [rng.choice(of[0], 90_000), rng.choice(of[2], 60_000), np.arange(n)]
    dst = [rng.choice(of[1], 90_000), rng.choice(of[2], 60_000), (np.arange(n) + np.choose(planted, (1, 2, 4, 4))) % n]
    for hubs, q in ((hubs_r, 0), (hubs_s, 2)):
        for h in hubs:
            from_q = of[q][of[q] != h]
            src += [rng.choice(from_q, HUB_EDGES), np.full(200, h)]
            dst += [np.full(HUB_EDGES, h), rng.choice(of[2] if q == 2 else of[3], 200)]
    b = planted.copy()
    b[hubs_r], b[hubs_s] = 0, 3
    return _G(n, np.concatenate(src), np.concatenate(dst)), np.concatenate([hubs_r, hubs_s]), b


# one launch for the whole pass; the degree groups' kernels (over 60,000 vertices)
@pytest.mark.parametrize("n", [2_000, 61_000])
@pytest.mark.parametrize("dl_fp32", [0, 1])
@pytest.mark.parametrize("dense_max_B", [1, 4096])
def test_hub_decisions_match_oracle(n, dl_fp32, dense_max_B):
    g, hubs, b = hub_graph(n)
    pm = P.Model(P.Graph(g.n, g.src, g.dst), 4, b, P.Params.default(seed=5, dl_fp32=dl_fp32, dense_max_B=dense_max_B))
    om = O.Model(O.Graph(g.n, g.src, g.dst), 4, b)
    left = np.zeros(hubs.size, bool)
    for sw in range(4):
        before = om.assignment()
        pm.sweep(sw)
        od = om.nodal_decide(5, sw, 3.0, nthreads=NT)
        margin = (od.s != before) & ((od.flags & 1) != 0) & \
                 (np.abs(od.lnu - od.logA) <= TOL * np.maximum(np.abs(od.logA), 1.0))
        got = pm.assignment()
        want = np.where(margin, got, od.b_new)
        assert np.array_equal(got, want), f"sweep {sw}: vertices {np.flatnonzero(got != want)[:5]}"
        left |= got[hubs] != b[hubs]
        om.set_b(4, got)
        check_blockmodel(pm, om)
    assert left.all()  # every hub's move was proposed and made


@pytest.mark.parametrize("movers_per_warp", [1, 2, 4])
def test_hub_in_a_batched_search_matches_oracle(movers_per_warp):
    g, _, _ = hub_graph(800, seed=1)
    ob, oB, odl, ons = O.partition(O.Graph(g.n, g.src, g.dst), O.Params(seed=2), nthreads=NT)
    pg = P.Graph(g.n, g.src, g.dst)
    opts = P.BatchOptions.default(max_B=1024, movers_per_warp=movers_per_warp)
    (b, B, dl, ns, _, _), = P.partition_batch([pg], P.Params.default(seed=2), opts)
    assert B == oB and ns == ons and np.array_equal(b, ob)
    assert dl == pytest.approx(odl, rel=1e-12)
