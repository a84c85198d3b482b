"""Bit-sliced sweep of rows that do not start on 16-byte boundaries (odd nx, or
a field on an 8-byte boundary) against the register sweep, which takes such
fields when the handle asks for the nibble variant: the same faces and windings,
whole numbers, element for element."""
import numpy as np
import pytest
import torch

import synth
from qtv_testutil import gpu_identify

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def handles():
    import paper_1911_12070_gb300 as qtv

    new, old = qtv.Qtv(0), qtv.Qtv(0)
    old.configure_sweep(variant=0)
    yield new, old
    new.close()
    old.close()


def _place(host, shift):
    """host on the device, `shift` elements past a 16-byte boundary, with NaN on
    both sides of the field."""
    buf = torch.full((host.size + 4,), complex(np.nan, np.nan), dtype=torch.complex64,
                     device="cuda")
    t = buf[2 + shift:2 + shift + host.size].view(host.shape)
    t.copy_(torch.from_numpy(host))
    return t


def _same(handles, psi):
    (ids, w, _), (ids0, w0, _) = gpu_identify(handles[0], psi), gpu_identify(handles[1], psi)
    assert np.array_equal(ids, ids0) and np.array_equal(w, w0)
    return len(ids)


# tile edges (124 columns; last tile of 1, of a stacked width, of a full one),
# band edges (16 rows), one plane, one row, the widest row
SHAPES = [(5, 17, 3), (3, 16, 125), (4, 33, 123), (6, 47, 127), (3, 18, 249), (2, 65, 253),
          (7, 1, 131), (1, 19, 77), (3, 20, 1023), (2, 17, 2047), (9, 50, 373), (300, 5, 35)]


@pytest.mark.parametrize("shift", [0, 1])
@pytest.mark.parametrize("shape", SHAPES)
def test_waves(handles, shape, shift):
    psi = synth.random_waves_numpy(shape, synth.wave_spec(sum(shape), 256, kmin=0.5, kmax=1.5))
    assert _same(handles, _place(psi, shift)) > 0


@pytest.mark.parametrize("shape", [(4, 18, 2), (3, 20, 124), (3, 33, 130), (4, 70, 256),
                                   (2, 17, 2048)])
def test_even_rows_off_the_boundary(handles, shape):
    psi = synth.random_waves_numpy(shape, synth.wave_spec(sum(shape), 256, kmin=0.5, kmax=1.5))
    assert _same(handles, _place(psi, 1)) > 0


@pytest.mark.parametrize("shape", [(5, 21, 37), (3, 40, 127), (4, 35, 251)])
@pytest.mark.parametrize("kind", ["ties", "signed zeros", "special", "tiny"])
def test_ties_zeros_and_nonfinite(handles, shape, kind):
    """Exactly antiparallel neighbours, zero nodes, -0.0, NaN and infinities,
    underflowing products: the exact path decides as the register sweep does."""
    rng = np.random.default_rng(sum(shape))
    re, im = rng.integers(-2, 3, (2,) + shape).astype(np.float32)
    if kind == "signed zeros":
        im = np.where(rng.random(shape) < 0.5, np.float32(-0.0), np.float32(0.0))
    if kind == "tiny":
        re, im = re * np.float32(3e-23), im * np.float32(2e-23)
    psi = (re + 1j * im).astype(np.complex64)
    if kind == "signed zeros":
        psi.imag[...] = im  # keeps the sign of zero
    if kind == "special":
        wave = synth.random_waves_numpy(shape, synth.wave_spec(7, 256))
        psi = np.where(rng.random(shape) < 0.01, psi, wave).astype(np.complex64)
        bad = rng.random(shape) < 0.002
        psi[bad] = rng.choice([complex(np.nan, 1), complex(np.inf, 0), complex(1, -np.inf),
                               complex(3e38, 3e38)], int(bad.sum()))
    for shift in (0, 1):
        _same(handles, _place(psi, shift))
