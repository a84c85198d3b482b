"""line_pieces of the binding: one pass for as many pieces as samples, and a result
that keeps no buffer of that size alive when there are few."""
import pytest
import torch

pytestmark = pytest.mark.gpu


def _chains(n, m):
    """n samples in chains of m: neighbours, degrees, components."""
    a = torch.arange(n, dtype=torch.int32)
    lo, hi = (a % m > 0), (a % m < m - 1) & (a + 1 < n)
    nbr = torch.full((n, 10), -1, dtype=torch.int32)
    nbr[:, 0] = torch.where(lo, a - 1, torch.where(hi, a + 1, -1))
    nbr[:, 1] = torch.where(lo & hi, a + 1, -1)
    return nbr.cuda(), (lo.int() + hi.int()).to(torch.uint8).cuda(), (a - a % m).contiguous().cuda()


class _Counted:
    def __init__(self, lib):
        self.lib, self.calls = lib, 0

    def __getattr__(self, name):
        f = getattr(self.lib, name)
        if name == "qtv_line_pieces":
            self.calls += 1
        return f


@pytest.mark.parametrize("m", [1, 2, 3, 5, 50])
def test_one_pass_and_no_large_buffer(monkeypatch, m):
    import paper_1911_12070_gb300 as qtv

    n = 30000
    q = qtv.Qtv(0)
    try:
        nbr, deg, comp = _chains(n, m)
        xyz = torch.rand((n, 3), device="cuda")
        counted = _Counted(qtv.lib())
        monkeypatch.setattr(qtv, "lib", lambda: counted)
        pieces, nodes = q.line_pieces(nbr, deg, comp, xyz)
        monkeypatch.undo()
        assert counted.calls == 1
        assert pieces.shape[0] == n // m and nodes.numel() == n
        assert pieces.untyped_storage().nbytes() <= 24 * (2 * (n // m) + 64)
        assert torch.equal(nodes.sort().values, torch.arange(n, dtype=torch.int32, device="cuda"))
    finally:
        q.close()


def test_capacities_one_short():
    # counts are complete, nothing is written past a capacity
    import ctypes

    import paper_1911_12070_gb300 as qtv

    n, m = 1000, 4
    q = qtv.Qtv(0)
    try:
        nbr, deg, comp = _chains(n, m)
        xyz = torch.rand((n, 3), device="cuda")
        for cap_p, cap_n in ((n // m, n), (n // m - 1, n), (n // m, n - 1), (0, 0)):
            pieces = torch.full((n, 24), 171, dtype=torch.uint8, device="cuda")
            nodes = torch.full((n + 1,), -7, dtype=torch.int32, device="cuda")
            counts = torch.zeros(2, dtype=torch.int64, device="cuda")
            p = [ctypes.c_void_p(t.data_ptr()) for t in (nbr, deg, comp, xyz)]
            rc = qtv.lib().qtv_line_pieces(
                q.h, n, None, *p, None, None, ctypes.c_void_p(pieces.data_ptr()) if cap_p else None,
                cap_p, ctypes.c_void_p(nodes.data_ptr()) if cap_n else None, cap_n,
                ctypes.c_void_p(counts.data_ptr()), None)
            assert rc == qtv.OK
            torch.cuda.synchronize()
            assert counts.tolist() == [n // m, n]
            assert (pieces[cap_p:] == 171).all() and (nodes[cap_n:] == -7).all()
            if (cap_p, cap_n) == (n // m, n):
                assert torch.equal(nodes[:n].cpu(), torch.arange(n, dtype=torch.int32))
    finally:
        q.close()
