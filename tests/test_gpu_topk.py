"""Top-k selection at the sizes where its two launches change shape, exact against a sort on
the host: fewer nodes than k, one element per thread, slices of several lanes, scores whose
slices' maxima say little (the list overflows and the last block selects by radix), heavy
ties, infinities and negative values."""
import numpy as np
import pytest

from oracle import linearization as lin

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def select():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.fail("CUDA device required for gpu tests")
    import paper_2004_03493_gb300 as esim
    esim.build()

    def run(scores, exclude, k):
        ids = torch.full((k,), -7, dtype=torch.int32, device="cuda")
        vals = torch.full((k,), -7.0, dtype=torch.float64, device="cuda")
        esim.esim_select_topk_static(torch.from_numpy(scores).cuda(), scores.size, exclude, k, ids, vals,
                                     torch.cuda.current_stream())
        return ids.cpu().numpy(), vals.cpu().numpy()

    return run


def _check(select, scores, exclude, k):
    ids, vals = select(scores, exclude, k)
    ids_ref, vals_ref = lin.topk(scores, k, exclude if exclude >= 0 else None)
    real = ids_ref.size if ids_ref.size < k else k
    assert np.array_equal(ids[:real], ids_ref[:real])
    assert np.array_equal(vals[:real], vals_ref[:real])
    assert np.all(ids[real:] == -1) and np.all(vals[real:] == 0.0)


def _scores(kind, n, rng):
    if kind == "equal":
        return np.full(n, 0.25)
    if kind == "ties":
        return np.round(rng.random(n) * 8) / 8
    if kind == "zeros":  # fewer positive scores than most k
        s = np.zeros(n)
        s[rng.integers(0, n, size=min(n, 37))] = rng.random(min(n, 37))
        return s
    if kind == "signed":
        s = rng.standard_normal(n)
        s[rng.integers(0, n, size=max(1, n // 100))] = np.inf
        s[rng.integers(0, n, size=max(1, n // 100))] = -np.inf
        return s
    return rng.random(n) ** 8


@pytest.mark.parametrize("kind", ["tail", "equal", "ties", "zeros", "signed"])
@pytest.mark.parametrize("n", [1, 2, 33, 1023, 1025, 4097, 70001, 400003, 1048577])
def test_sizes(select, n, kind):
    rng = np.random.default_rng(n)
    scores = _scores(kind, n, rng)
    for k, exclude in ((1, -1), (2, 0), (50, n - 1), (1000, -1), (4096, n // 2)):
        ids, _ = select(scores, exclude, k)
        assert exclude < 0 or exclude not in ids
        eligible = n - (1 if exclude >= 0 else 0)
        if eligible >= k:
            _check(select, scores, exclude, k)
        else:
            ids_ref, vals_ref = lin.topk(scores, max(eligible, 1), exclude if exclude >= 0 else None)
            got, vals = select(scores, exclude, k)
            assert np.array_equal(got[:eligible], ids_ref[:eligible])
            assert np.array_equal(vals[:eligible], vals_ref[:eligible])
            assert np.all(got[eligible:] == -1) and np.all(vals[eligible:] == 0.0)


@pytest.mark.parametrize("k", [100, 4096])
def test_large_scores_in_few_slices(select, k):
    """A quarter of k whole slices (32 consecutive ids in every stretch of one element per
    thread) hold the large scores: many more keys than the list holds reach the bound."""
    import torch
    threads = 2 * torch.cuda.get_device_properties(0).multi_processor_count * 1024
    n = 4 * threads - 5
    rng = np.random.default_rng(k)
    scores = rng.random(n)
    slices = rng.choice(threads // 32, size=k // 4, replace=False)
    lanes = (slices[:, None] * 32 + np.arange(32)).ravel()
    for row in range(4):
        at = lanes + row * threads
        at = at[at < n]
        scores[at] = 2.0 + rng.random(at.size)
    _check(select, scores, -1, k)
