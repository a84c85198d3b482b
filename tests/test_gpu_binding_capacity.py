"""The binding's first guesses of output sizes: a graph with more pieces than the
guess, a subset of the pieces, and no samples give what exact sizes give."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def q():
    import paper_1911_12070_gb300 as qtv

    h = qtv.Qtv(0)
    yield h
    h.close()


def _graph(adj):
    n = len(adj)
    nbr = np.full((n, 10), -1, np.int32)
    for a, s in enumerate(adj):
        nbr[a, :len(s)] = sorted(s)
    deg = np.array([len(s) for s in adj], np.uint8)
    comp, seen = np.zeros(n, np.int32), {}
    for a in range(n):
        todo = [a]
        while todo:
            u = todo.pop()
            if u not in seen:
                seen[u] = a
                todo += adj[u]
        comp[a] = seen[a]
    return [torch.from_numpy(t).cuda() for t in (nbr, deg, comp)]


@pytest.mark.parametrize("n", [0, 1, 600, 5000])
def test_lone_samples_exceed_the_guess(q, n):
    nbr, deg, comp = _graph([[] for _ in range(n)]) if n else [
        torch.zeros((0, 10), dtype=torch.int32, device="cuda"),
        torch.zeros(0, dtype=torch.uint8, device="cuda"),
        torch.zeros(0, dtype=torch.int32, device="cuda")]
    xyz = torch.rand((n, 3), device="cuda")
    pieces, nodes = q.line_pieces(nbr, deg, comp, xyz)
    assert tuple(pieces.shape) == (n, 24) and nodes.tolist() == list(range(n))
    curve, first, length = q.piece_curves(xyz, nodes, pieces)
    assert torch.equal(curve, xyz) and first.tolist() == list(range(n)) and not length.any()


def test_a_subset_of_the_pieces(q):
    n = 4000
    adj = [[v for v in (a - 1, a + 1) if v // 10 == a // 10 and 0 <= v < n] for a in range(n)]
    nbr, deg, comp = _graph(adj)
    xyz = torch.rand((n, 3), device="cuda")
    pieces, nodes = q.line_pieces(nbr, deg, comp, xyz)
    assert pieces.shape[0] == n // 10
    curve, first, length = q.piece_curves(xyz, nodes, pieces)
    some, sfirst, slength = q.piece_curves(xyz, nodes, pieces[7:9])
    a, b = int(first[7]), int(first[9])
    assert torch.equal(some, curve[a:b]) and torch.equal(slength, length[7:9])
    assert some.untyped_storage().nbytes() == some.numel() * 4
    # twice the same piece: more points than entries
    twice = torch.cat([pieces] * 3)
    many, _, mlength = q.piece_curves(xyz, nodes[:n], twice)
    assert torch.equal(many, torch.cat([curve] * 3)) and torch.equal(mlength, torch.cat([length] * 3))
