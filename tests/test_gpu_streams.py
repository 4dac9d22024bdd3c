"""Calls of one handle that lie on two streams, and of two handles in two threads: what each does
or leaves behind does not reach the other."""
import ctypes
import threading

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


@pytest.mark.parametrize("sync_between", [False, True])
def test_samples_on_two_streams(esim, oracle_walks, sync_between):
    """Two samples with buffers of their own, each of more chunks than the chip holds warps; with
    sync_between the handle's status block is reset while the first may still run."""
    import torch
    n, rp, col = synth.chung_lu(5000, 50000, gamma=2.1, seed=3)
    rng = np.random.default_rng(4)
    jobs = []
    for seed in (7, 8):
        R = rng.integers(0, 6000, size=n).astype(np.uint64)
        off = torch.from_numpy(np.concatenate([[0], np.cumsum(R)]).astype(np.uint64)).cuda()
        jobs.append((seed, off, torch.zeros(n, dtype=torch.uint64, device="cuda"),
                     torch.zeros(1, dtype=torch.uint64, device="cuda"), oracle_walks.walk_pairs(n, rp, col, R, C, seed)))
    streams = [torch.cuda.Stream() for _ in jobs]
    torch.cuda.synchronize()
    with esim.Graph(n, rp, col) as g:
        for _ in range(5):
            for stream, (seed, off, counts, steps, _ref) in zip(streams, jobs):
                g.set_stream(stream)
                if sync_between:
                    g.sync()
                g.sample(off, C, seed, counts, steps)
            torch.cuda.synchronize()
            for _seed, _off, counts, steps, (ref, ref_steps) in jobs:
                assert np.array_equal(counts.cpu().numpy(), ref)
                assert int(steps.cpu().numpy()[0]) == ref_steps
        g.set_stream(None)


def test_captured_sample(esim, oracle_walks):
    """A captured sample has no chunk counter: every block takes a fixed share."""
    import torch
    n, rp, col = synth.chung_lu(5000, 50000, gamma=2.1, seed=3)
    R = np.random.default_rng(6).integers(0, 700, size=n).astype(np.uint64)
    ref, ref_steps = oracle_walks.walk_pairs(n, rp, col, R, C, 5)
    off = torch.from_numpy(np.concatenate([[0], np.cumsum(R)]).astype(np.uint64)).cuda()
    counts = torch.zeros(n, dtype=torch.uint64, device="cuda")
    steps = torch.zeros(1, dtype=torch.uint64, device="cuda")
    stream = torch.cuda.Stream()
    with esim.Graph(n, rp, col) as g:
        g.set_stream(stream)
        g.sample(off, C, 4, counts, steps)
        torch.cuda.synchronize()
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph, stream=stream):
            g.sample(off, C, 5, counts, steps)
        for _ in range(2):
            counts.view(torch.int64).fill_(-1)
            torch.cuda.synchronize()
            graph.replay()
            torch.cuda.synchronize()
            assert np.array_equal(counts.cpu().numpy(), ref)
            assert int(steps.cpu().numpy()[0]) == ref_steps
        g.set_stream(None)


def test_selections_of_different_sizes_in_two_threads(esim):
    """k = 600 and k = 4096 need different amounts of shared memory for one kernel."""
    import torch
    n, rp, col = synth.erdos_renyi(9000, 30000, seed=2)
    scores = torch.rand(n, dtype=torch.float64, device="cuda")
    order = torch.sort(scores, descending=True).indices.to(torch.int32)
    failed = []

    def work(k):
        try:
            ids = torch.full((k,), -7, dtype=torch.int32, device="cuda")
            vals = torch.empty(k, dtype=torch.float64, device="cuda")
            with esim.Graph(n, rp, col) as g:
                for _ in range(4000):
                    g.select_topk(scores, -1, k, ids, vals)
                g.sync()
            assert torch.equal(ids, order[:k])
        except BaseException as e:  # reported by the main thread
            failed.append((k, e))

    torch.cuda.synchronize()
    threads = [threading.Thread(target=work, args=(k,)) for k in (600, 4096)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not failed


def test_calls_after_an_overlap_are_right(esim):
    """A forward and a reverse sweep of one handle on two streams share its scratch and may spoil
    each other (rows cut into pieces, other numbers of them in the two directions); what is called
    after them, one at a time, gives the same bits as before."""
    import torch
    n, rp, col = synth.chung_lu(20000, 400000, gamma=2.1, seed=2)
    L, k = 12, 700
    hist, bad = (torch.empty((L + 1) * n, dtype=torch.float64, device="cuda") for _ in range(2))
    s, bad_s = (torch.empty(n, dtype=torch.float64, device="cuda") for _ in range(2))
    pi = torch.empty(n, dtype=torch.float64, device="cuda")
    R = torch.empty(n, dtype=torch.uint64, device="cuda")
    off = torch.empty(n + 1, dtype=torch.uint64, device="cuda")
    ids = torch.empty(k, dtype=torch.int32, device="cuda")
    vals = torch.empty(k, dtype=torch.float64, device="cuda")
    dhat = torch.from_numpy(synth.uniform_diagonal(n, C)).cuda()
    streams = [torch.cuda.Stream() for _ in range(2)]
    torch.cuda.synchronize()
    with esim.Graph(n, rp, col) as g:
        def one_by_one():
            g.set_stream(streams[0])
            g.forward(3, C, L, hist)
            g.allocate(hist, L, 1e6, 0, pi, R, off)
            g.reverse(hist, L, C, dhat, s)
            g.select_topk(s, 3, k, ids, vals)
            g.sync()
            return [t.cpu().numpy().copy() for t in (hist, pi, R, off, s, ids, vals)]

        before = one_by_one()
        for _ in range(30):
            g.set_stream(streams[0])
            g.forward(3, C, L, bad)
            g.set_stream(streams[1])
            g.reverse(hist, L, C, dhat, bad_s)
            torch.cuda.synchronize()
            for a, b in zip(before, one_by_one()):
                assert np.array_equal(a, b)
        g.set_stream(None)


def test_a_refused_launch_does_not_fail_the_next_call(esim):
    """A sweep on a stream whose capture was invalidated is refused; the handle's next call, on a
    good stream, is not."""
    import torch
    n, rp, col = synth.erdos_renyi(300, 1500, seed=2)
    L = 3
    hist = torch.empty((L + 1) * n, dtype=torch.float64, device="cuda")
    off = torch.arange(n + 1, dtype=torch.int64, device="cuda").view(torch.uint64)
    counts = torch.zeros(n, dtype=torch.uint64, device="cuda")
    torch.cuda.synchronize()
    cudart = ctypes.CDLL(f"libcudart.so.{torch.version.cuda.split('.')[0]}")
    stream = torch.cuda.Stream()
    handle = ctypes.c_void_p(stream.cuda_stream)
    with esim.Graph(n, rp, col) as g:
        g.forward(1, C, L, hist)  # the workspace is there from here on
        g.sync()
        assert cudart.cudaStreamBeginCapture(handle, 2) == 0
        assert cudart.cudaStreamSynchronize(handle) != 0  # not allowed while capturing: the capture is invalid
        g.set_stream(stream)
        with pytest.raises(esim.EsimError):
            g.forward(1, C, L, hist)
        graph = ctypes.c_void_p()
        assert cudart.cudaStreamEndCapture(handle, ctypes.byref(graph)) != 0
        cudart.cudaGetLastError()
        g.set_stream(None)
        g.sample(off, C, 3, counts)
        g.sync()
