"""Vortex-node lists of tall thin grids, whose many (plane, sub-band) totals are scanned
tile by tile, by chunks of several tiles after a launch that sums those, or by one
block: ascending, complete and with the values of the dense field."""
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.mark.parametrize("shape", [(1, 3, 4), (2048, 9, 5), (2049, 12, 5), (131072, 3, 4), (131073, 3, 4),
                                   (140001, 19, 3), (4200001, 3, 3)])
def test_list_is_the_dense_field(shape):
    import paper_1911_12070_gb300 as qtv

    g = torch.Generator(device="cuda").manual_seed(shape[0])
    psi = torch.view_as_complex(torch.randn((*shape, 2), generator=g, device="cuda"))
    q = qtv.Qtv(0)
    try:
        ids, circ, dense = q.node_circulation(psi, capacity=psi.numel() // 4 + 64, dense=True)
        want = torch.nonzero((dense != 0).any(0).view(-1))[:, 0]
        assert torch.equal(ids, want)
        assert torch.equal(circ, dense.view(3, -1)[:, want].T)
    finally:
        q.close()
