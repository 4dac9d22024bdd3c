"""The sweeps' sliced rows at the lengths and node counts where their layout changes, against
the oracle: rows that just fit a lane or a piece (32, 64, 1024, 2048 entries), windows of
1024 rows with a remainder, pieces that are joined, hubs with positions of their own (more
than 8192 nodes, skewed uses), both row caps (below and above four million edges)."""
import numpy as np
import pytest

import synth
from oracle import linearization as lin

pytestmark = pytest.mark.gpu

C = 0.6
LENGTHS = [0, 1, 2, 7, 8, 9, 16, 31, 32, 33, 63, 64, 65, 100, 255, 257, 1023, 1024, 1025, 2047, 2048, 2049, 4097]


def _graph(n, transpose, seed, lengths=LENGTHS):
    """Row j has lengths[j % len] entries (at most n - 1) with distinct, skewed sources."""
    rng = np.random.default_rng(seed)
    w = (1.0 - rng.random(n)) ** -0.8
    order = np.argsort(-w)
    src, dst = [], []
    for j in range(n):
        d = min(lengths[j % len(lengths)], n - 1)
        if d == 0:
            continue
        draw = rng.choice(n, size=min(n, 2 * d + 8), p=w / w.sum())
        got = np.unique(draw[draw != j])[:d]
        if got.size < d:  # fill up with the heaviest nodes not drawn yet
            rest = order[(order != j) & ~np.isin(order, got)]
            got = np.concatenate([got, rest[:d - got.size]])
        src.append(got)
        dst.append(np.full(got.size, j))
    if not src:
        return synth.edges_to_in_csr(n, np.zeros(0, np.int64), np.zeros(0, np.int64))
    s, d = np.concatenate(src), np.concatenate(dst)
    return synth.edges_to_in_csr(n, d, s) if transpose else synth.edges_to_in_csr(n, s, d)


@pytest.mark.parametrize("transpose", [False, True])
@pytest.mark.parametrize("n", [1, 2, 33, 1023, 1025, 9001])
def test_forward_and_reverse(n, transpose):
    torch = pytest.importorskip("torch")
    import paper_2004_03493_gb300 as esim
    esim.build()
    n, rp, col = _graph(n, transpose, n)
    L, u = 6, (n - 1) // 2
    H = lin.hop_vectors(n, rp, col, u, C, L)
    D = synth.uniform_diagonal(n, C)
    s_ref = lin.reverse(n, rp, col, H, D, C)
    with esim.Graph(n, rp, col) as g:
        for _ in range(2):  # the second sweep finds the pieces' counts as the first left them
            hist = torch.full(((L + 1) * n,), float("nan"), dtype=torch.float64, device="cuda")
            s = torch.full((n,), float("nan"), dtype=torch.float64, device="cuda")
            g.forward(u, C, L, hist)
            g.reverse(hist, L, C, torch.from_numpy(D).cuda(), s)
            g.sync()
            assert np.max(np.abs(hist.view(L + 1, n).cpu().numpy() - H)) <= 1e-12
            assert np.max(np.abs(s.cpu().numpy() - s_ref)) <= 1e-12
        hist32 = torch.full(((L + 1) * n,), float("nan"), dtype=torch.float32, device="cuda")
        g.forward_f32(u, C, L, hist32)
        g.sync()
        got = hist32.view(L + 1, n).cpu().numpy().astype(np.float64)
        for l in range(L + 1):  # every stored pi^l is within (2 l + 2) u relative
            assert np.all(np.abs(got[l] - H[l]) <= (2 * l + 2) * 2.0 ** -24 * H[l] + 1e-30)


# Row lengths around a cap of 8, 16 and 32 and around its pieces (32 caps); the node counts make the
# loader choose that cap (more than 6080 rows above the next smaller one).
@pytest.mark.parametrize("transpose", [False, True])
@pytest.mark.parametrize("n,lengths", [
    (1500, [1, 7, 3, 8, 0, 9, 2, 255, 4, 256, 5, 257, 6, 513, 1, 1, 2, 2]),
    (7001, [10] * 60 + [15, 16, 17, 511] + [12] * 60 + [512, 513, 1025, 0]),
    (7001, [18] * 60 + [31, 32, 33, 1023] + [20] * 60 + [1024, 1025, 2049, 0]),
])
def test_row_caps(n, lengths, transpose):
    torch = pytest.importorskip("torch")
    import paper_2004_03493_gb300 as esim
    esim.build()
    n, rp, col = _graph(n, transpose, len(lengths), lengths)
    L, u = 5, n // 3
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
