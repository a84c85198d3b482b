"""Curve lengths at the ends of the FP32 range: distances whose squares overflow give
an infinite length, points that are not finite a NaN, and lengths of very large and
very small curves are those of a 64-bit sum."""
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


def _curve(q, pts, per):
    """One open piece through pts."""
    import paper_1911_12070_gb300 as qtv

    rec = np.zeros(1, qtv.PIECE_DTYPE)
    rec["count"] = len(pts)
    rec["comp_type"] = 1
    pieces = torch.from_numpy(rec.view(np.uint8).reshape(1, 24)).cuda()
    xyz = torch.tensor(np.asarray(pts, np.float32)).cuda()
    nodes = torch.arange(len(pts), dtype=torch.int32, device="cuda")
    curve, _, length = q.piece_curves(xyz, nodes, pieces, per)
    return curve.cpu().numpy(), float(length[0])


@pytest.mark.parametrize("per", [1, 2, 8])
@pytest.mark.parametrize("n", [2, 3, 40])
def test_overflow_is_infinite(q, per, n):
    x = np.arange(n, dtype=np.float64) * 1e25
    curve, length = _curve(q, np.stack([x, x * 0, x * 0], 1), per)
    assert np.isfinite(curve).all() and length == np.inf


@pytest.mark.parametrize("per", [1, 8])
def test_nan_point(q, per):
    pts = np.zeros((40, 3))
    pts[:, 0] = np.arange(40)
    pts[20, 1] = np.nan
    assert np.isnan(_curve(q, pts, per)[1])


@pytest.mark.parametrize("scale", [1e-12, 1.0, 1e15])
@pytest.mark.parametrize("per", [1, 8, 64])
def test_length_of_its_points(q, scale, per):
    rng = np.random.default_rng(per)
    curve, length = _curve(q, rng.standard_normal((300, 3)) * scale, per)
    exact = np.linalg.norm(np.diff(curve.astype(np.float64), axis=0), axis=1).sum()
    # FP32 distances: differences 1 unit, sum of squares 3 (half of both after the root: 2.5), root 1,
    # the sum rounded once to FP32 1
    assert abs(length - exact) <= 5 * 2.0 ** -24 * exact
