"""Dense records and reused scratch.  White noise fills every record of a segment, up
to the 32 steps of 31 columns that the narrow form of the expand pass orders through
shared memory and beyond them (the wide form); the face list has to be the one of the
other sweep.  Calls of different sizes through one handle find their counters, scan
tiles and segment totals zeroed whatever the call before left there."""
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


def _noise(shape, seed):
    g = torch.Generator().manual_seed(seed)
    return torch.view_as_complex(torch.randn((*shape, 2), generator=g)).cuda()


def _faces(q, psi):
    cap = 3 * psi.numel()
    ids = torch.zeros(cap, dtype=torch.int64, device="cuda")
    w = torch.zeros(cap, dtype=torch.int8, device="cuda")
    n = torch.zeros(1, dtype=torch.int64, device="cuda")
    q.identify_into(psi, ids, w, n)
    k = int(n)
    return ids[:k], w[:k]


@pytest.mark.parametrize("shape", [(3, 17, 34), (2, 16, 62), (5, 40, 990), (4, 33, 992), (4, 33, 994), (3, 20, 1100)])
def test_dense_records(shape):
    import paper_1911_12070_gb300 as qtv

    qtv.build()
    psi = _noise(shape, 7)
    q = qtv.Qtv(0)
    try:
        a = _faces(q, psi)
        q.configure_sweep(variant=0)
        b = _faces(q, psi)
    finally:
        q.close()
    assert a[0].numel() > psi.numel() // 2
    assert torch.equal(a[0], b[0]) and torch.equal(a[1], b[1])


def test_sizes_in_turn():
    import paper_1911_12070_gb300 as qtv

    qtv.build()
    fields = [_noise(s, i) for i, s in enumerate([(200, 530, 34), (4, 20, 64), (130, 513, 40), (2, 2, 34)])]
    q = qtv.Qtv(0)
    try:
        for psi in fields + fields[::-1]:
            f = qtv.Qtv(0)
            try:
                a, b = _faces(q, psi), _faces(f, psi)
            finally:
                f.close()
            assert torch.equal(a[0], b[0]) and torch.equal(a[1], b[1])
    finally:
        q.close()
