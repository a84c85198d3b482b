"""Box-mean reduction of a device count below the bound."""
import pytest

from test_gpu_reduce import _table, q  # noqa: F401  (q: the module's fixture)

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


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
