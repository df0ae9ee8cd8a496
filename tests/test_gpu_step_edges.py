"""The tabu step at the edges of its tiles: sequence lengths on either side of
each word count, searches that cross the 32-step blocks in which draws and key
offsets are renewed, the tie rule, and CTAs that run fewer warps than asked for
because the search's scratch would not fit.  All integers: bit-exact."""
import numpy as np
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


@pytest.mark.parametrize("fix_first", [False, True])
@pytest.mark.parametrize("N", [3, 8, 31, 32, 33, 64, 65, 96, 97, 128, 129, 160, 161, 192, 193, 255, 256])
def test_long_searches_equal_oracle(labs, orc, N, fix_first):
    """7 N + 65 steps from random and extreme starts (all +1 has the largest energy
    and ties everywhere): every move and energy of the trace equals the oracle's."""
    from paper_2504_00987_gb300 import workloads

    mi = 7 * N + 65
    starts = np.concatenate([workloads.random_sequences(N, 2, seed=N), workloads.sequence_edge_cases(N)])
    variant = labs.VARIANT_FIX_FIRST_SPIN if fix_first else 0
    d = torch.from_numpy(starts.view(np.int64)).cuda()
    plain = labs.tabu_run(d, N, 17, max_iter=mi, variant=variant)
    traced = labs.tabu_run(d, N, 17, max_iter=mi, variant=variant, trace_cap=mi)
    for key in ("best", "bestE", "steps"):
        assert torch.equal(plain[key], traced[key])
    for b in range(len(starts)):
        best, bestE, steps, tr = orc.tabu_run(starts[b], N, 17, b, 0, max_iter=mi, trace_cap=mi, variant=variant)
        assert int(traced["steps"][b]) == steps and int(traced["bestE"][b]) == bestE
        assert np.array_equal(traced["trace"][b, :steps].cpu().numpy(), tr)
        assert traced["best"][b].cpu().numpy().view(np.uint64).tolist() == [int(x) for x in best][: (N + 63) // 64]


@pytest.mark.parametrize("wps", [1, 2])
def test_ctas_of_fewer_warps(labs, wps):
    """Eight warps of K = 740 and N = 256 fit a CTA with their populations alone,
    not with the search's scratch: accepted, same results as one or two warps; a
    population that never fitted stays refused."""
    inst = [labs.make_instance(256, 740, seed=3, instance=i, max_steps=400) for i in range(5)]
    small = {"warps_per_block": wps, "blocks_per_sm": 1, "warps_per_seq": wps}
    big = {"warps_per_block": 8, "blocks_per_sm": 1, "warps_per_seq": wps}
    a, b = labs.mts_batch_run(inst, mapping=small), labs.mts_batch_run(inst, mapping=big)
    for x, y in zip(a, b):
        assert (x["E"], x["seq"], x["steps"]) == (y["E"], y["seq"], y["steps"])
    with pytest.raises(labs.LabsError):
        labs.mts_batch_run([labs.make_instance(256, 800, max_steps=400)], mapping=big)


def test_server_with_ctas_of_fewer_warps(labs):
    req = labs.make_instance(256, 740, seed=3, instance=1, max_steps=400)
    with labs.Server(max_slots=4, max_N=256, max_K=740, warps_per_block=8) as srv:
        t = srv.submit(req)
        got = None
        while got is None:
            got = srv.poll(t)
    alone = labs.mts_batch_run([req], mapping={"warps_per_block": 1, "blocks_per_sm": 1})[0]
    assert (got["E"], got["seq"], got["steps"]) == (alone["E"], alone["seq"], alone["steps"])
    with pytest.raises(labs.LabsError):
        labs.Server(max_slots=4, max_N=256, max_K=800, warps_per_block=8)
