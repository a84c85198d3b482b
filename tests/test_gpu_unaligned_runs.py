"""Bit-sliced sweep of unaligned rows over runs longer than its ring, over changes of
column within a CTA, in every tile shape, and on fields that take the exact edge test
in some or all planes, against the register sweep (which such fields take when a
handle is set to the nibble sweep): the same faces and windings, element for element.
A handle set to the bit-sliced sweep takes it for every row above 62 columns."""
import numpy as np
import pytest
import torch

import synth
from test_gpu_unaligned import SHAPES, _place, _same

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def register():
    import paper_1911_12070_gb300 as qtv

    q = qtv.Qtv(0)
    q.configure_sweep(variant=0)
    yield q
    q.close()


def _bits(warps=0, stages=0, ctas=0):
    import paper_1911_12070_gb300 as qtv

    q = qtv.Qtv(0)
    q.configure_sweep(variant=1, warps_per_tile=warps, stages=stages, ctas_per_sm=ctas)
    return q


def _waves(shape, seed=3):
    return synth.random_waves(shape, synth.wave_spec(seed, 64, kmin=0.3, kmax=0.9)).numpy()


def _field(shape, kind):
    rng = np.random.default_rng(sum(shape))
    psi = _waves(shape)
    if kind == "waves":
        return psi
    if kind == "noise":
        return (rng.standard_normal(shape) + 1j * rng.standard_normal(shape)).astype(np.complex64)
    if kind == "ties":  # small integers: equal and opposite neighbours, zeros
        return (rng.integers(-2, 3, shape) + 1j * rng.integers(-2, 3, shape)).astype(np.complex64)
    if kind == "slabs":  # planes of ties between smooth ones: the exact test on and off
        ties = _field(shape, "ties")
        for k in range(shape[0]):
            if (k // 5) % 3 == 1 or k % 29 == 0:
                psi[k] = ties[k]
        return psi
    if kind == "hole":  # zero outside a ball, signed zeros in the shell
        r2 = sum(((np.arange(n) - n / 2) / n).reshape([-1 if i == a else 1 for i in range(3)]) ** 2
                 for a, n in enumerate(shape))
        psi[r2 > 0.12] = 0
        psi.imag[(r2 > 0.1) & (r2 < 0.12)] = np.float32(-0.0)
        return psi
    if kind == "vanishing":  # amplitudes down to the smallest FP32 values
        return (psi * np.float32(10) ** rng.integers(-44, 3, shape).astype(np.float32)).astype(np.complex64)
    psi[rng.random(shape) < 1e-4] = np.nan
    psi[rng.random(shape) < 1e-4] = complex(np.inf, -np.inf)
    psi[rng.random(shape) < 1e-4] = complex(3e38, -3e38)
    return psi


@pytest.mark.parametrize("shape", [(140, 150, 253), (131, 97, 377)])
@pytest.mark.parametrize("kind", ["waves", "noise", "ties", "slabs", "hole", "vanishing", "special"])
@pytest.mark.parametrize("shift", [0, 1])
def test_long_runs(register, shape, kind, shift):
    q = _bits()
    try:
        assert _same((q, register), _place(_field(shape, kind), shift)) > 0
    finally:
        q.close()


@pytest.mark.parametrize("warps", [2, 4, 8])
@pytest.mark.parametrize("stages", [2, 3])
@pytest.mark.parametrize("ctas", [0, 1])
def test_tile_shapes(register, warps, stages, ctas):
    q = _bits(warps, stages, ctas)
    try:
        for shape, shift in (((90, 130, 253), 0), ((41, 97, 378), 1), ((200, 33, 65), 0), ((30, 70, 639), 1)):
            for kind in ("waves", "slabs"):
                assert _same((q, register), _place(_field(shape, kind), shift)) > 0
    finally:
        q.close()


@pytest.mark.parametrize("shape", [s for s in SHAPES if s[2] > 62] + [(4, 18, 65), (3, 20, 124), (5, 21, 67)])
@pytest.mark.parametrize("kind", ["waves", "ties", "vanishing", "special"])
def test_small_grids(register, shape, kind):
    # the edges of bands and tiles, which the default handle may leave to the register sweep
    q = _bits()
    try:
        for shift in (0, 1):
            _same((q, register), _place(_field(shape, kind), shift))
    finally:
        q.close()


@pytest.mark.parametrize("nx,shift", [(61, 0), (62, 1), (63, 0), (63, 1), (64, 1), (65, 0), (66, 1), (93, 0),
                                      (94, 1), (95, 0), (123, 1), (125, 0), (126, 1), (155, 0), (157, 1)])
@pytest.mark.parametrize("kind", ["slabs", "special"])
def test_narrow_rows(register, nx, shift, kind):
    q = _bits()
    try:
        assert _same((q, register), _place(_field((70, 65, nx), kind), shift)) > 0
    finally:
        q.close()


# on both sides of the rule of the default handle: rows of a band, columns of a tile
@pytest.mark.parametrize("shape", [(40, 7, 251), (40, 8, 251), (40, 16, 125), (40, 17, 125), (40, 33, 127),
                                   (40, 32, 127), (90, 70, 63), (90, 64, 63), (90, 70, 65), (30, 14, 1001),
                                   (30, 16, 1001)])
def test_default_handle(register, shape):
    import paper_1911_12070_gb300 as qtv

    q = qtv.Qtv(0)
    try:
        for shift in (0, 1):
            assert _same((q, register), _place(_field(shape, "slabs"), shift)) > 0
    finally:
        q.close()


def test_reserve_covers_both_alignments(register):
    # 17 rows of 126 columns: the staged sweep aligned, the register sweep 8 bytes off
    import paper_1911_12070_gb300 as qtv

    shape = (40, 17, 126)
    psi = _place(_field(shape, "waves"), 1)
    q = qtv.Qtv(0)
    try:
        cap = psi.numel()
        q.reserve(shape, cap)
        ids = torch.zeros(cap, dtype=torch.int64, device="cuda")
        w = torch.zeros(cap, dtype=torch.int8, device="cuda")
        n = torch.zeros(1, dtype=torch.int64, device="cuda")
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph):
            q.identify_into(psi, ids, w, n)
        graph.replay()
        torch.cuda.synchronize()
        ids0, w0, _ = register.identify(psi)
        k = int(n)
        assert torch.equal(ids[:k], ids0) and torch.equal(w[:k], w0)
    finally:
        q.close()
