"""Refinement at the lines of its dispatch: below 32 steps and above four samples a
lane one kernel does all of a call, else a second one takes up the searches that the
first leaves to a list, whose counters are zero again after each call.  A sample's
result is the same bits in all of them."""
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

SHAPE = (40, 52, 75)


@pytest.fixture(scope="module")
def setup():
    import paper_1911_12070_gb300 as qtv

    qtv.build()
    q = qtv.Qtv(0)
    nz, ny, nx = SHAPE
    g = torch.Generator().manual_seed(11)
    psi = torch.view_as_complex(torch.randn((nz, ny, nx, 2), generator=g) + 0.7).cuda()
    x0 = (torch.rand((100000, 3), generator=g) * torch.tensor([nx, ny, nz])).cuda()
    yield q, psi, x0
    q.close()


def _bits(r, sel=slice(None)):
    return [(v[sel].contiguous().view(torch.int32) if v.is_floating_point() else v[sel])
            for v in r.values()]


def _same(a, b):
    return all(torch.equal(u, v) for u, v in zip(a, b))


@pytest.mark.parametrize("n", [1, 31, 500, 24320, 24321, 97280, 97281, 100000])
def test_few_and_many_steps(setup, n):
    q, psi, x0 = setup
    x = x0[:n].contiguous()
    few, many = (q.refine_samples(psi, xyz0=x, max_iter=m) for m in (31, 32))
    ended = few["iters"] < 31
    assert _same(_bits(few, ended), _bits(many, ended))
    more = q.refine_samples(psi, xyz0=x, max_iter=33)
    ended = many["iters"] < 32
    assert _same(_bits(many, ended), _bits(more, ended))


def test_calls_in_turn_leave_the_counters(setup):
    q, psi, x0 = setup
    full = q.refine_samples(psi, xyz0=x0)
    for n, m in ((100000, 200), (7, 200), (3000, 5), (3000, 200), (100000, 5), (100000, 200)):
        r = q.refine_samples(psi, xyz0=x0[:n].contiguous(), max_iter=m)
        if m == 200:
            assert _same(_bits(r), _bits(full, slice(0, n)))


@pytest.mark.parametrize("n", [100, 100000])
@pytest.mark.parametrize("limit", [0, 1, 77])
def test_device_count(setup, n, limit):
    q, psi, x0 = setup
    ndev = torch.tensor([limit], dtype=torch.int64, device="cuda")
    r = q.refine_samples(psi, xyz0=x0[:n].contiguous(), n_dev=ndev)
    ref = q.refine_samples(psi, xyz0=x0[:100].contiguous())
    assert _same(_bits(r, slice(0, limit)), _bits(ref, slice(0, limit)))
