"""Sweeps of a graph below four million edges whose rows mostly lie between 32 and 64 entries: so many
that lanes take them, not warps (more than 24,320 warps at a cap of 32, a quarter fewer at 64)."""
import numpy as np
import pytest

import synth
from oracle import linearization as lin

pytestmark = pytest.mark.gpu

C = 0.6


@pytest.mark.parametrize("transpose", [False, True])
def test_rows_of_64(transpose):
    torch = pytest.importorskip("torch")
    import paper_2004_03493_gb300 as esim
    esim.build()
    n = 30_001
    rng = np.random.default_rng(3)
    lengths = np.resize([40] * 50 + [33, 48, 63, 64, 65, 2047, 2048, 2049, 0, 1], n)
    lengths[100:] = np.minimum(lengths[100:], 65)  # a few rows of one piece or two
    row = np.repeat(np.arange(n), lengths)
    start = np.concatenate([[0], np.cumsum(lengths)])
    step = rng.integers(1, 14, size=n)  # 14 * 2049 < n: distinct entries
    other = (row + 1 + rng.integers(0, n, size=n)[row] + (np.arange(row.size) - start[row]) * step[row]) % n
    n, rp, col = synth.edges_to_in_csr(n, row, other) if transpose else synth.edges_to_in_csr(n, other, row)
    assert col.size < 4_000_000
    L, u = 4, n // 3
    H = lin.hop_vectors(n, rp, col, u, C, L)
    D = synth.uniform_diagonal(n, C)
    s_ref = lin.reverse(n, rp, col, H, D, C)
    with esim.Graph(n, rp, col) as g:
        for _ in range(2):
            hist = torch.full(((L + 1) * n,), float("nan"), dtype=torch.float64, device="cuda")
            s = torch.full((n,), float("nan"), dtype=torch.float64, device="cuda")
            g.forward(u, C, L, hist)
            g.reverse(hist, L, C, torch.from_numpy(D).cuda(), s)
            g.sync()
            assert np.max(np.abs(hist.view(L + 1, n).cpu().numpy() - H)) <= 1e-12
            assert np.max(np.abs(s.cpu().numpy() - s_ref)) <= 1e-12
