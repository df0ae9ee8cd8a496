"""Populations at the limit of what a CTA's warps can keep: accepted or refused
by what 256 bytes a word beside the population would take, whatever the search's
scratch takes, and the same results as one warp (or pair) per CTA."""
import time

import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def labs():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__

    __graft_entry__.build()
    import paper_2504_00987_gb300 as labs

    return labs


def key(r):
    return (r["E"], r["seq"], r["steps"], r["generations"])


# warps_per_request 2: the links of the pairs take 128 bytes of a CTA beside the
# populations, so K = 672 (N = 256) and K = 907 (N = 192) miss eight warps by them
@pytest.mark.parametrize("N,K,wpr,accepted", [
    (256, 671, 2, True), (256, 672, 1, True), (256, 672, 2, True), (256, 673, 2, True), (192, 907, 2, True),
    (160, 1024, 2, True), (256, 749, 2, True), (256, 750, 1, True), (256, 750, 2, False), (256, 751, 1, False),
    (256, 751, 2, False), (192, 982, 2, True), (192, 983, 1, False)])
def test_servers(labs, N, K, wpr, accepted):
    opts = dict(max_slots=4, max_N=N, max_K=K, warps_per_block=8, warps_per_request=wpr)
    if not accepted:
        with pytest.raises(labs.LabsError):
            labs.Server(**opts)
        return
    reqs = [labs.make_instance(n, K, seed=3, instance=n, max_steps=300) for n in (N, 40)]
    with labs.Server(**opts) as srv:
        tickets = [srv.submit(r) for r in reqs]
        got, deadline = {}, time.time() + 60.0
        while len(got) < len(reqs):
            assert time.time() < deadline
            for t in tickets:
                if t not in got:
                    r = srv.poll(t)
                    if r is not None:
                        got[t] = r
        assert srv.stats()["failed"] == 0 and (wpr == 1 or srv.stats()["pair_quanta"] > 0)
    alone = labs.mts_batch_run(reqs, mapping={"warps_per_block": 1, "blocks_per_sm": 1})
    assert [key(got[t]) for t in tickets] == [key(r) for r in alone]


# the instance that takes most with the scratch is not always the one that decides acceptance
@pytest.mark.parametrize("wps", [1, 2])
@pytest.mark.parametrize("a,b,accepted", [((256, 749), (192, 981), True), ((256, 750), (192, 985), False),
                                          ((256, 740), (192, 1000), False)])
def test_mixed_batches(labs, a, b, accepted, wps):
    inst = [labs.make_instance(N, K, seed=4, instance=N, max_steps=300) for N, K in (a, b)]
    big = {"warps_per_block": 8, "blocks_per_sm": 1, "warps_per_seq": wps}
    if not accepted:
        with pytest.raises(labs.LabsError):
            labs.mts_batch_run(inst, mapping=big)
        return
    small = {"warps_per_block": wps, "blocks_per_sm": 1, "warps_per_seq": wps}
    assert [key(r) for r in labs.mts_batch_run(inst, mapping=big)] == \
        [key(r) for r in labs.mts_batch_run(inst, mapping=small)]
