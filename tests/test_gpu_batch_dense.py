"""Batched sweeps on dense graphs, whose pieces are longer than 64 entries, against the single-source
precision form; and that a dense graph's rows are not cut."""
import numpy as np
import pytest

import synth

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


def _regular(n, degree, extra, seed):
    """In-CSR: every node has `degree` in-neighbours (a random shift each), the first nodes have the
    lengths of `extra` instead."""
    rng = np.random.default_rng(seed)
    lengths = np.full(n, degree)
    lengths[:len(extra)] = extra
    rp = np.concatenate([[0], np.cumsum(lengths)]).astype(np.int64)
    row = np.repeat(np.arange(n), lengths)
    step = rng.choice([s for s in range(1, 200) if np.gcd(s, n) == 1], size=n)
    col = (row + 1 + rng.integers(0, n, size=n)[row] + (np.arange(rp[-1]) - rp[row]) * step[row]) % n
    return n, rp, col.astype(np.int32)


# pieces of 128 (mean degree 60) and 256 (110) entries; rows around one and two of them
@pytest.mark.parametrize("n,degree", [(18_001, 60), (20_011, 110)])
def test_long_pieces(esim, n, degree):
    n, rp, col = _regular(n, degree, [0, 1, 63, 64, 65, 127, 128, 129, 255, 256, 257, 511, 512, 513, 2049, 6000], degree)
    eps = 5e-2
    u = [6, 7, 10, 14, 17, n - 1]
    with esim.Graph(n, rp, col, kappa=4.0, precision=1) as g:
        want = [g.query(v, C, eps, 3) for v in u]
        L = g.stats()["L"]
        for extra in (0, 20, 50):
            for tile in (0, 1, 2):
                g.set_option("batch_tile", tile)
                s = g.query_batch(u + [n // 2] * extra, [eps] * (len(u) + extra), C, seed=3)
                for q in range(len(u)):
                    # an FP32 history on both sides: 2 L u relative each, on scores below 1
                    assert np.max(np.abs(s[q] - want[q])) <= 4 * L * 2.0 ** -24 / (1 - C)


def test_dense_graph_is_not_cut(esim):
    """Rows of 195 entries, all alike in both directions: a level is one launch."""
    n, degree = 20_000, 195
    shift = np.random.default_rng(1).choice(np.arange(1, n), size=degree, replace=False)
    rp = np.arange(n + 1, dtype=np.int64) * degree
    col = ((np.arange(n)[:, None] + shift) % n).astype(np.int32).ravel()
    with esim.Graph(n, rp, col, kappa=4.0) as g:
        g.query_batch(np.arange(16), [1e-2] * 16, C, 1)
        st = g.stats()
    assert st["launches"] <= 2 * st["L"] + 12, st
