"""The paper's depth rule where not every level's sets are kept (n above 45,000), and the number of
times it makes them.  Copies of one small graph side by side: a node's exploration stays in its
copy, so the oracle's counts on the small graph are every copy's."""
import numpy as np
import pytest

import synth
from oracle import alg3 as a3

pytestmark = pytest.mark.gpu

C = 0.6


@pytest.fixture(scope="module")
def esim():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.fail("CUDA device required for gpu tests")
    import paper_2004_03493_gb300 as pkg
    pkg.build()
    return pkg


def _small():
    """64 nodes: a sparse part whose supports keep growing, a denser one, nodes without in-edges."""
    rng = np.random.default_rng(5)
    src, dst = [], []
    for j in range(40):
        src += [(j + 1) % 40, (j + 7) % 40]
        dst += [j, j]
    for j in range(40, 58):
        for i in rng.choice(24, size=4, replace=False):
            src.append(40 + int(i))
            dst.append(j)
    return synth.edges_to_in_csr(64, np.array(src), np.array(dst))


# buffers in the rule's 4 GiB: 17 and every level kept, 13 (0..10 kept), 5 (0..2), 2 (none)
@pytest.mark.parametrize("copies", [40, 800, 1200, 2048])
def test_depths_with_levels_kept_or_made_twice(esim, copies):
    import torch
    n0, rp0, col0 = _small()
    E = a3.explored_edges(n0, rp0, col0, 16)
    n = n0 * copies
    rp = np.concatenate([[0], np.cumsum(np.tile(np.diff(rp0), copies))]).astype(np.int64)
    col = (np.tile(col0, copies) + np.repeat(np.arange(copies) * n0, col0.size)).astype(np.int32)
    rng = np.random.default_rng(copies)
    # 32 choices of R for every node of the small graph, by copy
    R0 = np.floor(10.0 ** rng.uniform(0, 6, size=(32, n0))).astype(np.uint64)
    R0[rng.random(R0.shape) < 0.2] = 0
    pick = rng.integers(0, 32, size=copies)
    for max_depth in (16, 6):
        want0 = np.array([[a3.paper_depth(E[:, k], int(R0[i, k]), C, max_depth) if R0[i, k] else 0 for k in range(n0)]
                          for i in range(32)], dtype=np.uint8)
        depth = torch.full((n,), 255, dtype=torch.uint8, device="cuda")
        with esim.Graph(n, rp, col) as g:
            for _ in range(2):
                g.alg3_paper_depth(torch.from_numpy(R0[pick].ravel().copy()).cuda(), C, max_depth, depth)
            g.sync()
        assert np.array_equal(depth.cpu().numpy(), want0[pick].ravel())
        assert len(np.unique(want0)) >= (10 if max_depth == 16 else 6)


def test_levels_are_made_once(esim):
    """On a skewed graph, where making a level is most of the rule's time, ten levels take no more
    than two and a half times four levels, and half as much again for the sums."""
    import time

    import torch
    n, rp, col = synth.chung_lu(2000, 16000, gamma=2.1, seed=3)
    E = a3.explored_edges(n, rp, col, 16)
    R = 100_000
    deepest = max(a3.paper_depth(E[:, k], R, C, 16) for k in range(n))
    assert deepest == 10
    depth = torch.empty(n, dtype=torch.uint8, device="cuda")
    with esim.Graph(n, rp, col) as g:
        def shortest(R, cap):
            R_d = torch.full((n,), R, dtype=torch.int64, device="cuda").view(torch.uint64)
            torch.cuda.synchronize()
            times = []
            for _ in range(6):
                start = time.perf_counter()
                g.alg3_paper_depth(R_d, C, cap, depth)
                g.sync()
                times.append(time.perf_counter() - start)
            return min(times[1:])

        four = shortest(10**15, 4)  # no node stops before the cap
        ten = shortest(R, 16)
    assert ten <= 1.5 * deepest / 4 * four
