"""Loads of a few entries more and fewer than what is copied with the small tables (65,536), of graphs
whose two CSRs have very different numbers of cut rows."""
import numpy as np
import pytest

import synth
from oracle import linearization as lin

pytestmark = pytest.mark.gpu

C = 0.6


@pytest.mark.parametrize("hubs", ["in", "out"])
@pytest.mark.parametrize("m", [65_535, 65_536, 65_537])
def test_entries_at_the_line(m, hubs):
    torch = pytest.importorskip("torch")
    import paper_2004_03493_gb300 as esim
    esim.build()
    n = 4001
    # ten rows of nearly all nodes, the others of the same few entries: distinct pairs, no loops
    row = np.repeat(np.arange(n), np.r_[np.full(10, 3900), np.full(n - 10, 7)])[:m]
    at = np.arange(row.size) - np.searchsorted(row, row)
    other = (row + 1 + at * (1 + (row >= 10) * (row % 500))) % n
    assert row.size == m
    n, rp, col = synth.edges_to_in_csr(n, other, row) if hubs == "in" else synth.edges_to_in_csr(n, row, other)
    assert col.size == m
    L, u = 3, 77
    H = lin.hop_vectors(n, rp, col, u, C, L)
    D = synth.uniform_diagonal(n, C)
    s_ref = lin.reverse(n, rp, col, H, D, C)
    with esim.Graph(n, rp, col) as g:
        hist = torch.full(((L + 1) * n,), float("nan"), dtype=torch.float64, device="cuda")
        s = torch.full((n,), float("nan"), dtype=torch.float64, device="cuda")
        g.forward(u, C, L, hist)
        g.reverse(hist, L, C, torch.from_numpy(D).cuda(), s)
        g.sync()
        assert np.max(np.abs(hist.view(L + 1, n).cpu().numpy() - H)) <= 1e-12
        assert np.max(np.abs(s.cpu().numpy() - s_ref)) <= 1e-12
