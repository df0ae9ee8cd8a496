"""The service with enough requests running that its CTAs have all the warps they
may have: every word class, none of them filling its last CTA."""
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


@pytest.mark.parametrize("warps", [2, 4, 8])
def test_ctas_of_several_warps(labs, orc, warps):
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    count = warps * sms // 2 + 40  # more than half of `warps` on every SM
    lengths = [(40, 64), (65, 96), (97, 128), (129, 160), (161, 192), (193, 256)]
    reqs = []
    for c, (lo, hi) in enumerate(lengths):
        share = (count // len(lengths) + c) | 1  # an odd number of requests in each class
        reqs += [labs.make_instance(lo + (7 * i) % (hi - lo + 1), 5 + i % 9, seed=6, instance=1000 * c + i, max_steps=6000)
                 for i in range(share)]
    with labs.Server(max_slots=len(reqs), max_N=256, max_K=16, warps_per_block=warps, quantum_steps=400) as srv:
        tickets = [srv.submit(r) for r in reqs]
        got, most, deadline = {}, 0, time.time() + 120.0
        while len(got) < len(reqs):
            assert time.time() < deadline
            most = max(most, srv.stats()["running"])
            for t in tickets:
                if t not in got:
                    r = srv.poll(t)
                    if r is not None:
                        got[t] = r
        assert srv.stats()["failed"] == 0
    assert 2 * most > warps * sms  # so some quantum ran CTAs of `warps` warps
    alone = labs.mts_batch_run(reqs, mapping={"warps_per_block": 1, "blocks_per_sm": 8})
    for t, r in zip(tickets, alone):
        g = got[t]
        assert (g["E"], g["seq"], g["steps"], g["generations"], g["status"]) == \
            (r["E"], r["seq"], r["steps"], r["generations"], r["status"])
    for i in range(0, len(reqs), max(1, len(reqs) // 8)):
        q = reqs[i]
        o, _, _ = orc.mts_run(orc.make_params(q.N, q.K, max_steps=q.max_steps), q.seed, q.instance)
        g = got[tickets[i]]
        assert (g["E"], g["steps"]) == (o["E"], o["steps"]) and g["seq"] == [int(x) for x in o["seq"]]
