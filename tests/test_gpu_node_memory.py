"""Workspace of the node form: staging follows the records that a grid can have (one
for nine rows of a column), not the capacity of the caller's lists, and a list as long
as the grid is filled completely."""
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


def test_staging_of_a_list_as_long_as_the_grid():
    import paper_1911_12070_gb300 as qtv

    n = 160
    g = torch.Generator(device="cuda").manual_seed(1)
    psi = torch.view_as_complex(torch.randn((n, n, n, 2), generator=g, device="cuda"))
    q = qtv.Qtv(0)
    try:
        ids = torch.zeros(psi.numel(), dtype=torch.int64, device="cuda")
        circ = torch.zeros((psi.numel(), 3), dtype=torch.int8, device="cuda")
        count = torch.zeros(1, dtype=torch.int64, device="cuda")
        q.node_circulation_into(psi[:2, :8, :8].contiguous(), ids, circ, count)
        torch.cuda.synchronize()
        free = torch.cuda.mem_get_info()[0]
        q.node_circulation_into(psi, ids, circ, count)
        torch.cuda.synchronize()
        grown = free - torch.cuda.mem_get_info()[0]
        # an eighth of the nodes (more than one for nine rows of 160) x 8/7 records of 20
        # bytes, 24 KB for each of 16 warps a multiprocessor, tables, allocation granules
        sms = torch.cuda.get_device_properties(0).multi_processor_count
        assert grown <= psi.numel() // 8 * 8 // 7 * 20 + sms * 16 * 24576 + (32 << 20)
        k = int(count)
        assert k > psi.numel() // 3 and (ids[1:k] > ids[:k - 1]).all() and (circ[:k] != 0).any(1).all()
        dense = torch.empty((3, n, n, n), dtype=torch.int8, device="cuda")
        q.node_circulation_into(psi, None, None, count, dense)
        assert k == int(count) == int((dense != 0).any(0).sum())
    finally:
        q.close()
