"""The sampler where few segments have pairs (a window is 32 pairs instead of 32 segments), bit for
bit against the C oracle, and that empty segments cost little."""
import numpy as np
import pytest

import synth

pytestmark = pytest.mark.gpu

C = 0.6


@pytest.fixture(scope="module")
def graph():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.fail("CUDA device required for gpu tests")
    import paper_2004_03493_gb300 as esim
    esim.build()
    data = synth.erdos_renyi(20_011, 60_000, seed=4)
    g = esim.Graph(*data)
    yield data, g
    g.close()


# every period-th node has pairs, from the first or the last one on; runs as long as a window, short
# ones, ones with a loop of their own in between, and stretches longer than a probe's reach (1024 segments)
@pytest.mark.parametrize("period", [2, 4, 5, 31, 32, 33, 64, 700, 5000])
@pytest.mark.parametrize("lengths", [[1], [7, 8], [20, 1, 1], [31, 32, 33], [1, 130, 2, 1, 1]])
def test_sparse_segments(graph, oracle_walks, period, lengths):
    import torch
    (n, rp, col), g = graph
    for first in (0, (n - 1) % period):
        R = np.zeros(n, dtype=np.uint64)
        at = np.arange(first, n, period)
        R[at] = np.resize(lengths, at.size)
        ref, ref_steps = oracle_walks.walk_pairs(n, rp, col, R, C, period)
        off = torch.from_numpy(np.concatenate([[0], np.cumsum(R)]).astype(np.uint64)).cuda()
        counts = torch.zeros(n, dtype=torch.uint64, device="cuda")
        steps = torch.zeros(1, dtype=torch.uint64, device="cuda")
        g.sample(off, C, period, counts, steps)
        g.sync()
        assert np.array_equal(counts.cpu().numpy(), ref)
        assert int(steps.cpu().numpy()[0]) == ref_steps


def test_empty_segments_cost_little():
    """One pair in every 64th node takes less than half the time of one in every node (a turn of a
    warp for every 32 segments took three quarters of it)."""
    import torch

    import paper_2004_03493_gb300 as esim
    n = 4_000_000
    rp = np.arange(n + 1, dtype=np.int64) * 2
    col = np.random.default_rng(1).integers(0, n, size=2 * n).astype(np.int32)
    stream = torch.cuda.Stream()
    counts = torch.zeros(n, dtype=torch.uint64, device="cuda")
    with esim.Graph(n, rp, col) as g:
        g.set_stream(stream)

        def shortest(period):
            R = np.zeros(n, dtype=np.int64)
            R[::period] = 1
            off = torch.from_numpy(np.concatenate([[0], np.cumsum(R)]).astype(np.uint64)).cuda()
            torch.cuda.synchronize()
            times = []
            for _ in range(8):
                start, end = (torch.cuda.Event(enable_timing=True) for _ in range(2))
                start.record(stream)
                g.sample(off, C, 3, counts)
                end.record(stream)
                end.synchronize()
                times.append(start.elapsed_time(end))
            return min(times[1:])

        every, sparse = shortest(1), shortest(64)
        g.set_stream(None)
    assert sparse < 0.5 * every
