"""Batches whose size is ragged against what a warp or a CTA takes at once, at
lengths on either side of each word count, against the oracle (exact)."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

NS = [3, 4, 16, 31, 32, 33, 47, 64, 65, 80, 96, 97, 128, 130, 161, 192, 224, 225, 256]


@pytest.fixture(scope="module")
def labs():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__

    __graft_entry__.build()
    import paper_2504_00987_gb300 as labs

    return labs


def sequences(N, B, dirty):
    """Random rows and the extreme ones; `dirty` sets the bits beyond N, which every call ignores."""
    from paper_2504_00987_gb300 import workloads

    a = np.concatenate([workloads.sequence_edge_cases(N), workloads.random_sequences(N, B, seed=B + N)])[:B]
    if dirty and N % 64:
        a = a.copy()
        a[:, -1] |= np.uint64((1 << 64) - (1 << (N % 64)))
    return a


def dev(a):
    return torch.from_numpy(np.ascontiguousarray(a).view(np.int64)).cuda()


@pytest.mark.parametrize("B", [1, 7, 33, 130])
@pytest.mark.parametrize("N", NS)
def test_skew_deviation(labs, orc, N, B):
    a = sequences(N, B, dirty=True)
    got = labs.skew_deviation_batch(dev(a), N).cpu().numpy()
    clean = sequences(N, B, dirty=False)
    for b in range(B):
        assert got[b] == orc.skew_deviation(clean[b], N)


@pytest.mark.parametrize("N", NS)
def test_energies_and_correlations(labs, orc, N):
    """Each way a batch is split: a warp a sequence one by one, four by four, a thread a
    sequence; the rows past the first few repeat them, so the oracle is asked once."""
    few = 37
    a = sequences(N, few, dirty=True)
    clean = sequences(N, few, dirty=False)
    ora = [orc.energy(x, N, with_C=True) for x in clean]
    E0 = np.array([e for e, _ in ora], dtype=np.int32)
    C0 = np.array([c for _, c in ora], dtype=np.int32)
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    nw = (N + 31) // 32
    for B in (1, few, 32 * sms, 32 * sms + 1, 8 * nw * nw * sms, 8 * nw * nw * sms + 3):
        rep = -(-B // few)
        d = dev(np.tile(a, (rep, 1))[:B])
        want = np.tile(E0, rep)[:B]
        assert np.array_equal(labs.energy_batch(d, N).cpu().numpy(), want)
        if B <= 32 * sms + 1:
            E, C = labs.energy_batch(d, N, with_C=True)
            assert np.array_equal(E.cpu().numpy(), want)
            assert np.array_equal(C.cpu().numpy(), np.tile(C0, (rep, 1))[:B])


@pytest.mark.parametrize("N", [3, 31, 64, 65, 128, 161, 192, 193, 224, 225, 256])
def test_energies_on_either_side_of_four_rows_a_warp(labs, orc, N):
    """The largest batch of one sequence a warp and the smallest of four, E with and
    without C; the rows past the first few repeat them, so the oracle is asked once."""
    few = 37
    a = sequences(N, few, dirty=True)
    ora = [orc.energy(x, N, with_C=True) for x in sequences(N, few, dirty=False)]
    E0 = np.array([e for e, _ in ora], dtype=np.int32)
    C0 = np.array([c for _, c in ora], dtype=np.int32)
    line = (192 if N > 192 else 48) * torch.cuda.get_device_properties(0).multi_processor_count
    for B in (line, line + 1, line + 3):
        rep = -(-B // few)
        d = dev(np.tile(a, (rep, 1))[:B])
        want = np.tile(E0, rep)[:B]
        E, C = labs.energy_batch(d, N, with_C=True)
        assert np.array_equal(E.cpu().numpy(), want)
        assert np.array_equal(C.cpu().numpy(), np.tile(C0, (rep, 1))[:B])
        assert np.array_equal(labs.energy_batch(d, N).cpu().numpy(), want)
