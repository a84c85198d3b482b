"""Face statistics on fields of small integers, where the FP32 products are
exact: zero-node, non-finite and ambiguous (exactly antiparallel edge) faces,
whole numbers equal to a numpy count."""
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


def _counts(psi):
    """(ambiguous, zero-node, non-finite) faces over the three orientations."""
    re, im = psi.real.astype(np.float64), psi.imag.astype(np.float64)
    fin = np.isfinite(re) & np.isfinite(im)
    zero = (re == 0) & (im == 0)
    re, im = np.where(zero | ~fin, 1.0, re), np.where(zero | ~fin, 0.0, im)
    tot = np.zeros(3, np.int64)
    for a, b in ((2, 1), (1, 0), (0, 2)):  # axes of the face: xy, yz, zx
        def at(t, da, db):
            s = [slice(None)] * 3
            s[a] = slice(da, t.shape[a] - 1 + da)
            s[b] = slice(db, t.shape[b] - 1 + db)
            return t[tuple(s)]

        loop = [(0, 0), (1, 0), (1, 1), (0, 1)]
        ok = np.logical_and.reduce([at(fin, *c) for c in loop])
        zer = np.logical_or.reduce([at(zero, *c) for c in loop])
        amb = np.zeros(ok.shape, bool)
        for c, d in zip(loop, loop[1:] + loop[:1]):
            dot = at(re, *c) * at(re, *d) + at(im, *c) * at(im, *d)
            crs = at(re, *c) * at(im, *d) - at(im, *c) * at(re, *d)
            amb |= (dot < 0) & (np.abs(crs) < 1e-4 * -dot)
        tot += [np.count_nonzero(amb & ok), np.count_nonzero(zer & ok), np.count_nonzero(~ok)]
    return tot


# edges of a warp's 31 columns, its 4 and a CTA's 32 rows, a chunk's 16 planes
@pytest.mark.parametrize("shape", [(1, 1, 1), (1, 40, 33), (16, 4, 31), (17, 5, 32), (18, 33, 63),
                                   (33, 32, 62), (15, 70, 1), (2, 1, 95), (5, 31, 257)])
@pytest.mark.parametrize("kind", ["dense", "rare"])
def test_integer_fields(q, shape, kind):
    rng = np.random.default_rng(sum(shape))
    re, im = rng.integers(-3, 4, (2,) + shape)
    if kind == "rare":  # most (plane, warp) pairs pass the screen
        calm = rng.random(shape) < 0.995
        re, im = np.where(calm, 2, re), np.where(calm, 1, im)
    psi = (re + 1j * im).astype(np.complex64)
    bad = rng.random(shape) < 0.003
    psi[bad] = rng.choice([complex(np.nan, 1), complex(np.inf, 2), complex(1, -np.inf)],
                          int(bad.sum()))
    _, _, st = q.identify(torch.from_numpy(psi).cuda(), stats=True)
    got = [st["ambiguous"], st["zero_node_faces"], st["nonfinite_faces"]]
    assert got == _counts(psi).tolist()
