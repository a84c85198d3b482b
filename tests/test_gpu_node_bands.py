"""Node form from psi at the edges of its work split: bands of 18 rows in two
sub-bands of 9, 30 columns a warp, z chunks, and segments with more records than a
warp holds in registers (every lane a vortex node); against the oracle's ring
circulation on unflagged rings, and list against dense field."""
import numpy as np
import pytest

import synth
from test_gpu_nodeform import _check, q  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("shape", [(3, 17, 29), (4, 18, 30), (5, 19, 31), (3, 27, 60), (6, 28, 61),
                                   (3, 36, 62), (12, 9, 33), (3, 3, 2048), (40, 20, 35)])
def test_edges_of_the_split(q, shape):  # noqa: F811
    _check(q, synth.random_waves_numpy(shape, synth.wave_spec(sum(shape), 256, kmin=0.5, kmax=1.5)))


@pytest.mark.parametrize("shape", [(5, 20, 300), (4, 40, 1000)])
def test_dense_noise(q, shape):  # noqa: F811
    rng = np.random.default_rng(sum(shape))
    psi = (rng.standard_normal(shape) + 1j * rng.standard_normal(shape)).astype(np.complex64)
    _check(q, psi)
