"""Top-k selection of scores that have an order by id: the lists, exact against a sort on the host,
and that the order costs nothing (slices that hold neighbours together select from most of the
scores in one block, 30 to 150 times slower)."""
import math

import numpy as np
import pytest

from oracle import linearization as lin

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def esim():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.fail("CUDA device required for gpu tests")
    import paper_2004_03493_gb300 as pkg
    pkg.build()
    return pkg


def _select(esim, scores, k):
    """(ids, scores, median microseconds) of 15 selections."""
    import torch
    dev = torch.from_numpy(scores).cuda()
    ids = torch.full((k,), -7, dtype=torch.int32, device="cuda")
    vals = torch.full((k,), -7.0, dtype=torch.float64, device="cuda")
    times = []
    for _ in range(15):
        start, end = (torch.cuda.Event(enable_timing=True) for _ in range(2))
        start.record()
        esim.esim_select_topk_static(dev, scores.size, -1, k, ids, vals, torch.cuda.current_stream())
        end.record()
        end.synchronize()
        times.append(1e3 * start.elapsed_time(end))
    return ids.cpu().numpy(), vals.cpu().numpy(), float(np.median(times))


def _pattern(kind, n, rng):
    s = rng.random(n) ** 8
    if kind == "ascending":
        return np.sort(s)
    if kind == "descending":
        return np.sort(s)[::-1].copy()
    if kind == "decay":  # around one id
        return np.exp(-np.abs(np.arange(n) - n // 2) / 5000.0)
    if kind == "few":  # fewer positive scores than k: the rest tie in id order
        s = np.zeros(n)
        s[rng.integers(0, n, size=37)] = rng.random(37)
        return s
    if kind == "community":
        s *= 1e-3
        s[n // 3:n // 3 + 5000] += rng.random(5000)
        return s
    if kind == "equal":
        return np.full(n, 0.25)
    if kind == "column":  # one column of a grid of 1024 ids a row
        s[5::1024] += 1.0
        return s
    return s


@pytest.mark.parametrize("k", [50, 1000, 4096])
@pytest.mark.parametrize("n", [100_003, 1_048_573])
def test_order_by_id(esim, n, k):
    rng = np.random.default_rng(n + k)
    _, _, random_us = _select(esim, _pattern("random", n, rng), k)
    for kind in ("ascending", "descending", "decay", "few", "community", "equal", "column"):
        scores = _pattern(kind, n, rng)
        ids, vals, us = _select(esim, scores, k)
        ids_ref, vals_ref = lin.topk(scores, k, None)
        assert np.array_equal(ids, ids_ref) and np.array_equal(vals, vals_ref), kind
        assert us <= 3.0 * random_us + 20.0, (kind, us, random_us)


@pytest.mark.parametrize("k", [100, 3000])
def test_large_scores_against_the_dealing(esim, k):
    """The large scores lie in the places of a few blocks, whose slices' maxima bound little: more
    keys reach the bound than the list holds, and the last block selects by radix."""
    import torch
    n = 1_048_573
    groups = -(-n // 32)
    A = int(groups * 0.6180339887498949) + 1
    while math.gcd(A, groups) != 1:
        A += 1
    place = np.arange(groups, dtype=np.int64) * A % groups
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    blocks = sms if 4 * k <= 32 * sms else 2 * sms
    few = k // 64 if k > 1000 else 1  # 32 slices each: fewer than k
    q = np.flatnonzero(place % (32 * blocks) < 32 * few)
    rng = np.random.default_rng(k)
    scores = rng.random(n)
    at = (32 * q[:, None] + np.arange(32)).ravel()
    at = at[at < n]
    assert at.size > 2 * k + 1024
    scores[at] = 2.0 + rng.random(at.size)
    ids, vals, _ = _select(esim, scores, k)
    ids_ref, vals_ref = lin.topk(scores, k, None)
    assert np.array_equal(ids, ids_ref) and np.array_equal(vals, vals_ref)
