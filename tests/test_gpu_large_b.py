"""The decision pass above 2048 blocks against the oracle: rows at the edges
of the degree classes and their tables, blocks whose rows are read through
and blocks whose rows are probed, dense and sparse.  Labels are compared bit
for bit outside the margin band, then M, degrees and DL."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

import oracle as O  # noqa: E402
import paper_2305_18663_gb300 as P  # noqa: E402
from synth.dcsbm import random_labels  # noqa: E402
from test_gpu_parity import _G, untraced_sweeps_vs_oracle  # noqa: E402

pytestmark = pytest.mark.gpu


def _graph(n, seed):
    """low degrees, a few vertices of every class's first and last degree,
    repeats (counts above 1) and self-loops"""
    rng = np.random.default_rng(seed)
    src, dst = [rng.integers(0, n, 2 * n)], [rng.integers(0, n, 2 * n)]
    v = 0
    for k in (30, 32, 33, 126, 128, 129, 510, 512, 513, 1598, 1600, 1601, 2500):
        for _ in range(4):
            ends = rng.integers(0, n, k // 2)
            src += [np.full(ends.size, v), rng.choice(n, k - ends.size)]
            dst += [ends, np.full(k - ends.size, v)]
            v += 1
    src += [np.arange(40), np.full(50, 3)]
    dst += [np.arange(40), np.full(50, 17)]
    return _G(n, np.concatenate(src), np.concatenate(dst))


@pytest.mark.parametrize("m_form", ["sparse", "dense"])
@pytest.mark.parametrize("B", [2049, 6000])
@pytest.mark.parametrize("skew", [False, True])
def test_pass_matches_oracle(B, m_form, skew):
    if m_form == "dense" and B > 4096:
        pytest.skip("dense models hold 4096 blocks here")
    g = _graph(9000, seed=B)
    b = random_labels(g.n, B, seed=1)
    if skew:  # half the vertices in ten blocks: their rows are long
        b[::2] = np.arange(b[::2].size) % 10
    untraced_sweeps_vs_oracle(g, B, b, P.Graph(g.n, g.src, g.dst), O.Graph(g.n, g.src, g.dst), m_form, sweeps=3,
                              seed=2, min_moves=1000)


@pytest.mark.parametrize("B", [2049, 6000])
def test_exact_form_decides_alike(B):
    g = _graph(9000, seed=B + 1)
    b = random_labels(g.n, B, seed=3)
    pg = P.Graph(g.n, g.src, g.dst)
    models = [P.Model(pg, B, b, P.Params.default(seed=4, dl_fp32=f, dense_max_B=d)) for f in (0, 1) for d in (1, 16384)]
    for sw in range(3):
        stats = [m.sweep(sw) for m in models]
        for m, st in zip(models[1:], stats[1:]):
            assert np.array_equal(m.assignment(), models[0].assignment())
            assert (st.n_moves, st.n_accepted, st.n_entries) == (stats[0].n_moves, stats[0].n_accepted, stats[0].n_entries)
