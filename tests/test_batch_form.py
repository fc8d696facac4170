"""The form of the batching form's persistent launches: a cluster of CTAs per
search while few searches are unfinished, one CTA per search else; and the
tuner's sample, which runs in the form of the batch it stands for."""
import pytest

import paper_2305_18663_gb300 as P


@pytest.mark.parametrize("sms,server,limits", [
    (152, False, {8: 17, 4: 34, 2: 68}), (152, True, {8: 9, 4: 19, 2: 38}),
    (132, False, {8: 14, 4: 29, 2: 59}), (1, False, {8: 0, 4: 0, 2: 0}),
])
def test_ctas_per_search(sms, server, limits):
    # the largest number of searches that still fits each form's share
    for ctas, most in limits.items():
        if most:
            assert P.sbp_search_form_check(most, sms, server) == ctas
            assert P.sbp_search_form_check(most + 1, sms, server) == ctas // 2
    assert P.sbp_search_form_check(10_000, sms, server) == 1
    with pytest.raises(P.SbpError):
        P.sbp_search_form_check(-1, sms, server)


@pytest.mark.gpu
def test_tuning_sample_runs_in_the_form_of_its_batch():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from synth.dcsbm import dcsbm

    pgs = []
    for i in range(80):
        n = 200 + 3 * i
        g = dcsbm(n, 8 * n, 4, 2.5, 1, 60, 4.0, seed=i)
        pgs.append(P.Graph(g.n, g.src, g.dst))
    prm = P.Params.default(seed=1)

    def launches(call):
        a = P.sbp_search_launches()
        call()
        b = P.sbp_search_launches()
        return b[0] - a[0], b[1] - a[1]

    # ten graphs run on clusters, and so does a tuner's sample of all of them
    assert launches(lambda: P.partition_batch(pgs[:10], prm))[0] == 0
    one, clusters = launches(lambda: P.autotune_batch(pgs[:10], prm, sample=10))
    assert one == 0 and clusters > 0
    # a sample of eight out of eighty stands for a batch with a CTA per search
    one, clusters = launches(lambda: P.autotune_batch(pgs, prm, sample=8))
    assert one > 0 and clusters == 0
