"""Where the one-launch pass and the one-launch commit end: on both sides of
each line the call takes the form it should (seen in the number of kernels it
launches) and gives what the general kernels give.  Labels, counts, degrees,
statistics and DL are compared exactly.  The forms of the batch kernels (CTA
shapes, register budgets and sub-batches by size) decide alike."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

import paper_2305_18663_gb300 as P  # noqa: E402
from synth.dcsbm import random_labels  # noqa: E402
from test_gpu_small import _same  # noqa: E402

pytestmark = pytest.mark.gpu


def _launches(call):
    before = P.sbp_kernel_launches()
    call()
    return P.sbp_kernel_launches() - before


def _graph(n, extra, seed):
    """every vertex with two edges out and two in; then `extra`: None, "hub"
    (one vertex with 300 edges more), "mid" (64 with 40 more) or a number of
    random edges in all"""
    rng = np.random.default_rng(seed)
    v = np.arange(n)
    src, dst = [v, v], [(v + 1) % n, (v + n // 3) % n]
    if extra == "hub":
        src, dst = src + [np.zeros(300, np.int64)], dst + [rng.integers(0, n, 300)]
    elif extra == "mid":
        src, dst = src + [np.repeat(np.arange(64), 40)], dst + [rng.integers(64, n, 64 * 40)]
    elif extra:
        src, dst = src + [rng.integers(0, n, extra - 2 * n)], dst + [rng.integers(0, n, extra - 2 * n)]
    return P.Graph(n, np.concatenate(src).astype(np.int32), np.concatenate(dst).astype(np.int32))


@pytest.mark.parametrize("n,extra,B,one", [
    (5_000, None, 1022, True), (5_001, None, 100, False), (2_500, None, 1023, True), (2_501, None, 1023, False),
    (22_000, "hub", 100, True), (22_001, "hub", 100, False), (10_000, "hub", 1023, True), (10_001, "hub", 1023, False),
    (40_000, "mid", 100, True), (40_001, "mid", 100, False), (20_000, "mid", 1023, True), (20_001, "mid", 1023, False),
    (20_000, 1 << 19, 100, True), (20_001, 1 << 19, 100, False),
    (6_000, 1 << 19, 1023, True), (6_001, 1 << 19, 1023, False),
    (2_000, 3 << 19, 100, True), (2_000, (3 << 19) + 1, 100, False),
])
def test_pass_form_and_result(n, extra, B, one):
    pg = _graph(n, extra, seed=n)
    b = random_labels(n, B, seed=1)
    for dl_fp32 in (1, 0):
        prm = P.Params.default(seed=4, dl_fp32=dl_fp32)
        whole, parts = P.Model(pg, B, b, prm), P.Model(pg, B, b, prm)
        for sw in range(2):
            k = _launches(lambda: P.sbp_nodal_decide(whole.h, sw, 0, n))
            if sw > 0:  # (the first pass also makes the block-labelled rows)
                assert (k == 1) == one, k
            for lo, hi in ((0, n // 3), (n // 3, n)):
                P.sbp_nodal_decide(parts.h, sw, lo, hi)
            a, c = P.sbp_commit(whole.h), P.sbp_commit(parts.h)
            assert a.n_moves > 0 and a.as_dict() | {"n_recheck": 0} == c.as_dict() | {"n_recheck": 0}
        _same(whole, parts)


@pytest.mark.parametrize("n,e", [(1_500, 3_000), (65_536, 131_072), (65_537, 131_074), (20_000, 1 << 19),
                                 (20_000, (1 << 19) + 1)])
@pytest.mark.parametrize("B", [2, 256, 257])
def test_commit_form_and_result(n, e, B):
    pg = _graph(n, None if e == 2 * n else e, seed=n)
    b = random_labels(n, B, seed=5)
    one = P.Model(pg, B, b, P.Params.default(seed=6))
    full = P.Model(pg, B, b, P.Params.default(seed=6, full_rebuild=1))
    small = n <= 65_536 and e <= 1 << 19 and B <= 256
    rng = np.random.default_rng(7)

    def sweep(sw, stats=True):
        a, c = one.sweep(sw, stats=stats), full.sweep(sw)
        if stats:
            assert a.as_dict() | {"n_recheck": 0} == c.as_dict() | {"n_recheck": 0}
        _same(one, full)

    sweep(0)  # random labels: many moves
    sweep(1)
    sweep(2, stats=False)
    # labels set from outside, few of them changed, many, few again; the pass
    # after each finds the form of the commit before it
    for sw, frac in ((3, 0.003), (4, 0.9), (5, 0.003)):
        lab = one.assignment()
        pick = rng.random(n) < frac
        lab[pick] = random_labels(n, B, seed=sw)[pick]
        k = _launches(lambda: P.sbp_set_assignment(one.h, B, lab))
        # one kernel lists the changes, one commits them
        assert (k == 2) == (small and (frac < 0.1 or n < 2_000)), k
        P.sbp_set_assignment(full.h, B, lab)
        _same(one, full)
        sweep(sw)


def _device_graph(n, e, seed):
    gen = torch.Generator(device="cuda").manual_seed(seed)
    src = torch.randint(0, n, (e,), generator=gen, device="cuda", dtype=torch.int32)
    return P.Graph(n, src, torch.randint(0, n, (e,), generator=gen, device="cuda", dtype=torch.int32))


# rows on both sides of 32 edges; B at the edges of the sub-batches' range, of
# the CTA shapes and of the kernels; then the exact form's other budgets
@pytest.mark.parametrize("n,e,Bs", [
    (30_000, 600_000, (63, 64, 320, 321, 460, 461, 1500, 1550, 2048)),
    (1 << 18, 4_400_000, (50,)),
    (300_000, 10 << 20, (100, 101)),
])
def test_batch_kernel_forms_decide_alike(n, e, Bs):
    pg = _device_graph(n, e, seed=n)
    for B in Bs:
        b = random_labels(n, B, seed=B)
        models = [P.Model(pg, B, b, P.Params.default(seed=2, dl_fp32=f, dense_max_B=d)) for f in (1, 0) for d in (4096, 1)]
        parts = P.Model(pg, B, b, P.Params.default(seed=2))  # its movers come from lists
        for sw in range(2):
            stats = [m.sweep(sw) for m in models]
            for lo, hi in ((0, n // 3), (n // 3, n)):
                P.sbp_nodal_decide(parts.h, sw, lo, hi)
            stats.append(P.sbp_commit(parts.h))
            assert stats[0].n_moves > n // 2 and stats[0].n_accepted > 0
            for m, st in zip(models[1:] + [parts], stats[1:]):
                assert np.array_equal(m.assignment(), models[0].assignment())
                assert (st.n_moves, st.n_accepted, st.n_entries) == \
                       (stats[0].n_moves, stats[0].n_accepted, stats[0].n_entries)
                assert st.dl_after == stats[0].dl_after


# Labels set from outside, more of them changed than one launch commits but
# less than three times as many: the commit of the pass after is asked about
# its own moves, and takes the form that they call for.
@pytest.mark.parametrize("B", [8, 64, 256])
def test_commit_form_after_labels_set(B):
    n, m = 20_000, 40_000
    pg = _graph(n, None, seed=n)  # four edge ends a vertex
    b = random_labels(n, B, seed=5)
    one = P.Model(pg, B, b, P.Params.default(seed=6))
    full = P.Model(pg, B, b, P.Params.default(seed=6, full_rebuild=1))
    for sw in range(20):
        one.sweep(sw), full.sweep(sw)
    lab = one.assignment()
    pick = np.random.default_rng(7).random(n) < 0.6
    lab[pick] = random_labels(n, B, seed=8)[pick]
    assert _launches(lambda: P.sbp_set_assignment(one.h, B, lab)) > 2
    P.sbp_set_assignment(full.h, B, lab)
    for sw in range(20, 30):
        P.sbp_nodal_decide(one.h, sw, 0, n)
        got = []
        k = _launches(lambda: got.append(P.sbp_commit(one.h)))
        c = full.sweep(sw)
        assert got[0].as_dict() | {"n_recheck": 0} == c.as_dict() | {"n_recheck": 0}
        acc = got[0].n_accepted
        load = acc + (acc // 10 if 16 * acc <= m else m // 80) + B * B // 64
        assert (k == 1) == (load <= 6000 + 32_000 // B), (sw, k, load)
        _same(one, full)


# the most blocks of the one-launch commit of a pass, few vertices moving
@pytest.mark.parametrize("B,one_launch", [(257, True), (512, True), (513, False)])
def test_commit_form_at_many_blocks(B, one_launch):
    n = 1_500
    pg = _graph(n, None, seed=n)
    b = random_labels(n, B, seed=5)
    one = P.Model(pg, B, b, P.Params.default(seed=6))
    full = P.Model(pg, B, b, P.Params.default(seed=6, full_rebuild=1))
    for sw in range(4):
        P.sbp_nodal_decide(one.h, sw, 0, n)
        got = []
        k = _launches(lambda: got.append(P.sbp_commit(one.h)))
        assert (k == 1) == one_launch, k
        assert got[0].as_dict() | {"n_recheck": 0} == full.sweep(sw).as_dict() | {"n_recheck": 0}
        _same(one, full)


# more than 1022 blocks, rows in the second and in the third group
@pytest.mark.parametrize("n,one", [(20_001, True), (40_000, True), (40_001, False)])
def test_pass_form_with_all_groups(n, one):
    rng = np.random.default_rng(n)
    v = np.arange(n)
    mid, far = np.repeat(np.arange(64), 40), np.repeat(np.arange(64, 128), 200)
    src = np.concatenate([v, v, mid, far])
    dst = np.concatenate([(v + 1) % n, (v + n // 3) % n, rng.integers(128, n, mid.size + far.size)])
    pg = P.Graph(n, src.astype(np.int32), dst.astype(np.int32))
    b = random_labels(n, 1_023, seed=1)
    prm = P.Params.default(seed=4)
    whole, parts = P.Model(pg, 1_023, b, prm), P.Model(pg, 1_023, b, prm)
    for sw in range(2):
        k = _launches(lambda: P.sbp_nodal_decide(whole.h, sw, 0, n))
        if sw > 0:
            assert (k == 1) == one, k
        for lo, hi in ((0, n // 3), (n // 3, n)):
            P.sbp_nodal_decide(parts.h, sw, lo, hi)
        a, c = P.sbp_commit(whole.h), P.sbp_commit(parts.h)
        assert a.n_moves > 0 and a.as_dict() | {"n_recheck": 0} == c.as_dict() | {"n_recheck": 0}
    _same(whole, parts)
