"""The walk-pair sampler's ways of taking work, bit for bit against the C oracle: segment
lengths around a warp (32), the shortest run with a loop of its own (128) and a chunk
(256), stretches of empty segments longer than a search round, one segment that holds
nearly every pair, nodes without in-edges, and the pair number's carry into its high word."""
import numpy as np
import pytest

import synth

pytestmark = pytest.mark.gpu

C = 0.6
EDGES = [0, 1, 2, 31, 32, 33, 63, 64, 65, 127, 128, 129, 255, 256, 257, 511, 513]


def _pattern(name, n, rng):
    R = np.zeros(n, dtype=np.uint64)
    if name == "ones":
        R[:] = 1
    elif name == "edges":
        R[:] = rng.choice(EDGES, size=n)
    elif name == "gaps":  # empty stretches of more than 1024 segments, at both ends too
        R[[1, n // 2, n // 2 + 1, n - 2]] = [5, 129, 3, 40]
    elif name == "heavy":
        R[:] = rng.integers(0, 3, size=n)
        R[n // 3] = 700_001
    elif name == "last":
        R[n - 1] = 1000
    elif name == "one":
        R[n // 2] = 1
    return R


@pytest.fixture(scope="module", params=["dangling", "chung_lu"])
def graph(request):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.fail("CUDA device required for gpu tests")
    import paper_2004_03493_gb300 as esim
    esim.build()
    data = synth.with_dangling(4001, 20000, seed=5) if request.param == "dangling" else synth.chung_lu(
        5000, 50000, gamma=2.1, seed=3)
    g = esim.Graph(*data)
    yield data, g
    g.close()


@pytest.mark.parametrize("with_depth", [False, True])
@pytest.mark.parametrize("pattern", ["none", "one", "ones", "edges", "gaps", "heavy", "last"])
def test_sampler_work_shapes(graph, oracle_walks, pattern, with_depth):
    import torch
    (n, rp, col), g = graph
    rng = np.random.default_rng(11)
    R = _pattern(pattern, n, rng)
    depth = rng.integers(0, 9, size=n).astype(np.uint8) if with_depth else np.zeros(n, dtype=np.uint8)
    off = np.concatenate([[0], np.cumsum(R)]).astype(np.uint64)
    ref, ref_steps = oracle_walks.walk_pairs_depth(n, rp, col, R, depth, C, 9)
    off_d, depth_d = torch.from_numpy(off).cuda(), torch.from_numpy(depth).cuda()
    counts = torch.zeros(n, dtype=torch.uint64, device="cuda")
    steps = torch.zeros(1, dtype=torch.uint64, device="cuda")
    for _ in range(2):  # the second launch finds the chunk counter as the first one left it
        counts.view(torch.int64).fill_(-1)
        g.sample_depth(off_d, depth_d if with_depth else None, C, 9, counts, steps)
        g.sync()
        assert np.array_equal(counts.cpu().numpy(), ref)
        assert int(steps.cpu().numpy()[0]) == ref_steps


def test_pair_number_carry(oracle_walks):
    """Pairs 2^32 - 100 .. 2^32 + 99 of one node: the difference of two launches' counts against
    the walks played out with the oracle's generator."""
    torch = pytest.importorskip("torch")
    import paper_2004_03493_gb300 as esim
    n, rp, col = synth.complete_digraph(5)
    k, c, seed, lo, hi = 2, 0.2, 6, 2**32 - 100, 2**32 + 100
    T = oracle_walks.threshold(c)
    ref = 0
    for r in range(lo, hi):
        a = b = k
        t = 0
        while True:
            ctr = np.array([[r & 0xFFFFFFFF, r >> 32, k, t]], dtype=np.uint32)
            w = [int(x) for x in oracle_walks.philox(ctr, seed)[0]]
            if not (w[0] < T and w[2] < T):
                ref += 1
                break
            for word, d in ((w[1], 4), (w[3], 4)):  # 4 divides 2^32: no word is rejected
                assert (word * d & 0xFFFFFFFF) >= 2**32 % d
            a, b = col[rp[a] + (w[1] * 4 >> 32)], col[rp[b] + (w[3] * 4 >> 32)]
            if a == b:
                break
            t += 1
    counts = []
    with esim.Graph(n, rp, col) as g:
        for total in (lo, hi):
            off = torch.tensor([0, 0, 0, total, total, total], dtype=torch.int64, device="cuda").view(torch.uint64)
            out = torch.zeros(n, dtype=torch.uint64, device="cuda")
            g.sample(off, c, seed, out)
            g.sync()
            counts.append(int(out.cpu().numpy()[k]))
    assert counts[1] - counts[0] == ref
