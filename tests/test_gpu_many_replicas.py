"""Seven and eight words with as many replicas as take the kernels of up to 255
registers and one more, which takes those of 128: launches and resumed slices, the
whole space and skew-symmetric sequences.  All integers: bit-exact."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

K, GENERATIONS = 6, 3


@pytest.fixture(scope="module")
def labs():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__

    __graft_entry__.build()
    import paper_2504_00987_gb300 as labs

    return labs


@pytest.mark.parametrize("N,skew", [(193, False), (200, False), (224, False), (225, False), (256, False),
                                    (201, True), (223, True), (225, True), (255, True)])
def test_replicas_on_either_side_of_eight_per_sm(labs, orc, N, skew):
    few = 8 * torch.cuda.get_device_properties(0).multi_processor_count
    variant = labs.VARIANT_SKEW if skew else 0

    def params(generations, mod=labs):
        return mod.make_params(N, K, max_generations=generations, variant=variant)

    a = labs.mts_launch(params(GENERATIONS), 5, 100, few)
    b = labs.mts_launch(params(GENERATIONS), 5, 100, few + 1)
    assert torch.equal(a, b[:few])
    results = labs.decode_results(b, N, 100)
    for r in (0, 1, few // 2, few - 1, few):
        o, _, _ = orc.mts_run(params(GENERATIONS, orc), 5, 100 + r)
        g = results[r]
        assert (g["E"], g["steps"], g["generations"]) == (o["E"], o["steps"], o["generations"])
        assert g["seq"] == [int(x) for x in o["seq"]]
    for R in (few, few + 1):
        state = torch.zeros(R * labs.mts_state_bytes(N, K), dtype=torch.uint8, device="cuda")
        labs.mts_resume(params(1), 5, 100, R, state, resume=False)
        c = labs.mts_resume(params(GENERATIONS), 5, 100, R, state, resume=True)
        assert np.array_equal(c.cpu().numpy(), b[:R].cpu().numpy())
