"""Callers on several threads whose launches of one kernel take different amounts
of shared memory: none may disturb another's launch.  Every run here is bounded
and every failure is a host-side error code."""
import threading
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


def together(*jobs):
    """Runs the jobs on a thread each; their exceptions."""
    errors = []

    def run(job):
        try:
            job()
        except Exception as e:  # reported by the caller's assertion
            errors.append(repr(e))

    threads = [threading.Thread(target=run, args=(j,)) for j in jobs]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    return errors


def serve(srv, reqs):
    deadline = time.time() + 120.0
    out = {}
    tickets = [srv.submit(r) for r in reqs]
    while len(out) < len(tickets):
        assert time.time() < deadline
        for t in tickets:
            if t not in out:
                r = srv.poll(t)
                if r is not None:
                    out[t] = r
        time.sleep(0.002)
    return [(out[t]["E"], out[t]["seq"], out[t]["steps"]) for t in tickets]


def test_busy_and_idle_servers(labs):
    """One server with more than two requests an SM runs CTAs of four warps, the
    other, of the same options, CTAs of one: thousands of quanta side by side."""
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    opts = dict(max_slots=2 * sms + 16, max_N=256, max_K=512, warps_per_block=4, quantum_steps=1)
    many = [labs.make_instance(256, 4, seed=1, instance=i, max_generations=300, max_iter=16)
            for i in range(2 * sms + 6)]
    one = [labs.make_instance(256, 4, seed=2, instance=0, max_generations=3000, max_iter=16)]
    got = {}
    with labs.Server(**opts) as a, labs.Server(**opts) as b:
        errors = together(lambda: got.update(many=serve(a, many)), lambda: got.update(one=serve(b, one)))
        assert errors == []
        assert a.stats()["quanta"] > 100 and b.stats()["quanta"] > 1000
    for name, reqs in (("many", many), ("one", one)):
        alone = labs.mts_batch_run(reqs, mapping={"warps_per_block": 1, "blocks_per_sm": 4})
        assert got[name] == [(r["E"], r["seq"], r["steps"]) for r in alone]


def test_launches_of_large_and_small_populations(labs):
    def launches(K, resume):
        P = labs.make_params(256, K, max_generations=0)
        s = torch.cuda.Stream()
        out = torch.zeros((1, 8), dtype=torch.int64, device="cuda")
        state = torch.zeros(labs.mts_state_bytes(256, K), dtype=torch.uint8, device="cuda")
        for _ in range(20_000):
            if resume:
                labs.mts_resume(P, 1, 0, 1, state, resume=False, out=out, stream=s)
            else:
                labs.mts_launch(P, 1, 0, 1, out=out, stream=s)
        s.synchronize()

    for resume in (False, True):
        assert together(lambda: launches(1024, resume), lambda: launches(2, resume)) == []


def test_batches_of_large_and_small_ctas(labs):
    def batches(K, wpb):
        inst = [labs.make_instance(256, K, max_generations=0)]
        for _ in range(500):
            with labs.Batch(inst, mapping={"warps_per_block": wpb, "blocks_per_sm": 1}) as b:
                b.launch()
                assert b.results()[0]["generations"] == 0

    assert together(lambda: batches(600, 8), lambda: batches(2, 1)) == []
