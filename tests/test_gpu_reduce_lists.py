"""Box-mean reduction with more edges between clusters than the edge lists hold
(they hold one per node), in all or in the first passes, and at the edges of a
block of nodes: against the oracle's graph.box_reduce, bit for bit."""
import numpy as np
import pytest

from oracle import graph
from test_gpu_reduce import _check, q  # noqa: F401  (q: the module's fixture)

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [1, 2, 255, 257, 2000])
@pytest.mark.parametrize("degree", [1, 3, 10])
@pytest.mark.parametrize("extent", [10.0, 40.0])
def test_random_graphs(q, n, degree, extent):  # noqa: F811
    rng = np.random.default_rng(n + degree)
    pos = rng.random((n, 3)) * extent
    adj = [set() for _ in range(n)]
    for _ in range(n * degree // 2):
        a, b = (int(v) for v in rng.integers(0, n, 2))
        if a != b and len(adj[a]) < 10 and len(adj[b]) < 10:
            adj[a].add(b)
            adj[b].add(a)
    _check(q, graph.Graph(pos, np.zeros_like(pos), adj), 4.0)
