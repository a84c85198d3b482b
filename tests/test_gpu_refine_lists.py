"""A sample's refinement does not depend on the list that it is in: searches longer
than a patience that grows with the list go to a second kernel with sixteen lanes
each, so short lists, long lists and single samples take different paths with the
same arithmetic.  Results are compared bit by bit."""
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

SHAPE = (44, 61, 83)


@pytest.fixture(scope="module")
def setup():
    import paper_1911_12070_gb300 as qtv

    qtv.build()
    q = qtv.Qtv(0)
    nz, ny, nx = SHAPE
    g = torch.Generator().manual_seed(5)
    # noise over a plane wave: zeros, box boundaries and searches of many halvings
    psi = torch.randn((nz, ny, nx, 2), generator=g) + 0.7
    psi = torch.view_as_complex(psi).cuda()
    x0 = torch.rand((120000, 3), generator=g) * (torch.tensor([nx, ny, nz]) + 1.0) - 1.0
    x0 = x0.cuda()
    full = q.refine_samples(psi, xyz0=x0)
    yield q, psi, x0, full
    q.close()


@pytest.mark.parametrize("n,start", [(1, 7), (31, 100), (33, 3000), (129, 50000), (5000, 9), (60000, 60000)])
def test_same_bits_in_any_list(setup, n, start):
    q, psi, x0, full = setup
    out = q.refine_samples(psi, xyz0=x0[start:start + n].contiguous())
    assert out.keys() == full.keys()
    for k, v in out.items():
        a, b = v, full[k][start:start + n]
        if a.is_floating_point():
            a, b = a.view(torch.int32), b.contiguous().view(torch.int32)
        assert torch.equal(a, b), k


@pytest.mark.parametrize("max_iter", [1, 3, 1000])
def test_step_limits(setup, max_iter):
    q, psi, x0, _ = setup
    long = q.refine_samples(psi, xyz0=x0, max_iter=max_iter)
    assert int(long["iters"].max()) <= max_iter
    short = q.refine_samples(psi, xyz0=x0[:300].contiguous(), max_iter=max_iter)
    for k, v in short.items():
        a, b = v, long[k][:300]
        if a.is_floating_point():
            a, b = a.view(torch.int32), b.contiguous().view(torch.int32)
        assert torch.equal(a, b), k


def test_second_launch(setup):
    # more than four samples a lane: the searches put off are taken up twice
    q, psi, x0, full = setup
    out = q.refine_samples(psi, xyz0=x0.repeat(6, 1))
    for k, v in out.items():
        for i in range(6):
            a, b = v[i * 120000:(i + 1) * 120000], full[k]
            if a.is_floating_point():
                a, b = a.view(torch.int32), b.view(torch.int32)
            assert torch.equal(a, b), (k, i)
