"""What a load finds out about a graph: repeated in-edges are neighbours in the out-edge CSR, and equal
neighbours of two rows are not repeated."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

ENOTSUP = -6


def _csr(n, edges):
    """In-CSR of (source, target) pairs as given, repeated ones kept."""
    edges = sorted(edges, key=lambda e: (e[1], e[0]))
    rp = np.zeros(n + 1, dtype=np.int64)
    for _, j in edges:
        rp[j + 1] += 1
    return n, np.cumsum(rp), np.array([i for i, _ in edges], dtype=np.int32)


# (edges, whether one is repeated)
GRAPHS = {
    "empty": ([], False),
    "one": ([(0, 1)], False),
    "star": ([(i, 0) for i in range(1, 40)], False),  # every row of the out-CSR is (0,)
    "star_and_one_twice": ([(i, 0) for i in range(1, 40)] + [(17, 0)], True),
    "last_and_first_alike": ([(0, 3), (0, 5), (1, 5), (1, 7), (4, 7)], False),
    "last_row_twice": ([(0, 3), (39, 2), (39, 2)], True),
    "first_row_twice": ([(0, 3), (0, 3), (39, 2)], True),
    "self_loop_twice": ([(5, 5), (5, 5)], True),
    "gaps": ([(3, 9), (20, 9), (30, 9)], False),  # rows without out-edges between them
}


@pytest.mark.parametrize("name", list(GRAPHS))
def test_repeated_in_edges(name):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.fail("CUDA device required for gpu tests")
    import paper_2004_03493_gb300 as esim
    esim.build()
    edges, repeated = GRAPHS[name]
    with esim.Graph(*_csr(40, edges)) as g:
        if repeated:
            with pytest.raises(esim.EsimError) as e:
                g.set_option("alg3", 1)
            assert e.value.status == ENOTSUP
        else:
            g.set_option("alg3", 1)
        assert abs(g.query(0, 0.6, 1e-2, 1)[0] - 1.0) <= 1e-2
