"""Box-mean reduction of a device count far below the bound (the launches then have
blocks that no pass needs) on graphs with more than two edges a node and boxes
that merge little, so that a pass hands on more edges than it had nodes: against
the oracle's graph.box_reduce, bit for bit, alone and beside another stream's work."""
import numpy as np
import pytest

from oracle import graph
from test_gpu_reduce import _check, _table, q  # noqa: F401  (q: the module's fixture)

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


def _graph(nn, seed):
    rng = np.random.default_rng(seed)
    pos = (rng.random((nn, 3)) * 40).astype(np.float32).astype(np.float64)
    adj = [set() for _ in range(nn)]
    for a, b in rng.integers(0, nn, (nn * 3, 2)):
        if a != b and len(adj[a]) < 10 and len(adj[b]) < 10:
            adj[a].add(int(b))
            adj[b].add(int(a))
    assert sum(map(len, adj)) >= 4 * nn
    return graph.Graph(pos, np.zeros_like(pos), adj)


@pytest.mark.parametrize("busy", [False, True])
@pytest.mark.parametrize("nn,n,box", [(1, 5000, 2.0), (255, 70000, 6.0), (1000, 100000, 2.0),
                                      (3000, 40000, 0.5), (3000, 400000, 8.0)])
def test_device_count_far_below_the_bound(q, nn, n, box, busy):  # noqa: F811
    g = _graph(nn, nn + n) if nn > 1 else graph.Graph(np.ones((1, 3)), np.zeros((1, 3)), [set()])
    red, lab, _, passes = graph.box_reduce(g, box)
    nbr, deg = _table(g.adj + [set()] * (n - nn), 10)
    xyz = torch.zeros((n, 3), device="cuda")
    xyz[:nn] = torch.from_numpy(g.pos.astype(np.float32))
    ndev = torch.tensor([nn], dtype=torch.int64, device="cuda")
    side = torch.cuda.Stream()
    m = torch.rand((2048, 2048), device="cuda")
    torch.cuda.synchronize()
    for _ in range(5 if busy else 1):
        if busy:
            with torch.cuda.stream(side):
                for _ in range(10):
                    m = (m @ m).clamp_(-1, 1)
        label, reps, pos, p = q.box_reduce(nbr, deg, xyz, box=box, n_dev=ndev)
        assert p == passes and np.array_equal(label.cpu().numpy()[:nn], lab)
        assert np.array_equal(reps.cpu().numpy(), np.unique(lab))
        assert np.array_equal(pos.cpu().numpy(), red.pos)
    torch.cuda.synchronize()


@pytest.mark.parametrize("extra", [-1, 0, 1])
@pytest.mark.parametrize("box", [0.25, 6.0])
def test_two_edges_a_node(q, extra, box):  # noqa: F811
    # the edge lists hold two a node: one less, as many and one more between clusters
    n = 700
    rng = np.random.default_rng(n + extra)
    pos = (rng.random((n, 3)) * 40).astype(np.float32).astype(np.float64)
    edges = {(i, (i + d) % n) for i in range(n) for d in (1, 2)}
    if extra < 0:
        edges.discard((5, 6))
    if extra > 0:
        edges.add((3, 400))
    adj = [set() for _ in range(n)]
    for a, b in edges:
        adj[a].add(b)
        adj[b].add(a)
    assert sum(map(len, adj)) == 2 * (2 * n + extra)
    _check(q, graph.Graph(pos, np.zeros_like(pos), adj), box)


def test_entries_past_the_device_count_are_no_clusters(q):  # noqa: F811
    # the memory of the labels still holds those of a call on all nodes
    n, nn = 50000, 700
    nbr, deg = _table([set()] * n, 10)
    xyz = torch.rand((n, 3), device="cuda") * 40
    full = q.box_reduce(nbr, deg, xyz)
    assert full[1].numel() == n
    del full
    ndev = torch.tensor([nn], dtype=torch.int64, device="cuda")
    _, reps, pos, _ = q.box_reduce(nbr, deg, xyz, n_dev=ndev)
    assert reps.tolist() == list(range(nn)) and pos.shape == (nn, 3)
