"""Training step of the learned locator on tcgen05 at batches whose 64-row chunks
divide into few splits of the weight gradients (then computed 64 columns a block)
or many, and whose last 128-row tile is half full, against the mma.sync layer kernels (the same BF16 operands,
FP32 accumulation in another order)."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu

SIZES = [("W1", 256 * 128), ("b1", 256), ("W2", 256 * 256), ("b2", 256), ("W3", 768), ("b3", 3)]


@pytest.fixture(scope="module")
def q():
    import paper_1911_12070_gb300 as qtv

    h = qtv.Qtv(0)
    yield h
    h.close()


@pytest.mark.parametrize("n", [64, 128, 64 * 15, 64 * 17, 64 * 32, 64 * 71, 64 * 100, 128 * 153])
def test_gradients_equal_the_layer_kernels(q, n):
    gen = torch.Generator(device="cuda").manual_seed(n)
    x = torch.randn((n, 128), generator=gen, device="cuda").bfloat16().view(torch.int16)
    t = torch.rand((n, 3), generator=gen, device="cuda")
    q.locator_init(n)
    got = {}
    for path in (1, 0):
        q.locator_set_tensor_path(path)
        g, loss = q.locator_gradients(x, t)
        got[path] = g.cpu().numpy().astype(np.float64), float(loss)
    q.locator_set_tensor_path(1)
    assert got[1][1] == pytest.approx(got[0][1], rel=1e-4)
    at = 0
    for name, size in SIZES:
        a, b = got[1][0][at:at + size], got[0][0][at:at + size]
        at += size
        # bound of the existing comparison of the two paths
        assert np.linalg.norm(a - b) < 1e-2 * np.linalg.norm(b), name
    again, _ = q.locator_gradients(x, t)
    assert np.array_equal(again.cpu().numpy().astype(np.float64), got[1][0])
    # the step uses these gradients: first Adam step, p - lr sign(g) where g is not tiny
    p0, _, _ = q.locator_get()
    q.locator_train_step(x, t, 1e-3)
    p1, adam, _ = q.locator_get()
    assert np.allclose(adam[:p1.size], 0.1 * got[1][0], rtol=1e-5, atol=1e-30)
    assert np.allclose(p1 - p0, -1e-3 * got[1][0] / (np.abs(got[1][0]) + 1e-8), atol=2e-6)
