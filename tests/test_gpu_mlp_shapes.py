"""Forward and backward kernels of the proposer at the sizes where their tiles
end: one row, one short of / past a tile, one chunk and many,
hidden widths that are no multiple of a tile."""
import numpy as np
import pytest

from oracle import mlp as omlp

pytestmark = pytest.mark.gpu

# sums of n * H FP32 products, added in tiles and chunks: a few 2^-24 sqrt(n H) of the largest term
SIZES = [(1, 16), (2, 1), (63, 128), (65, 33), (1024, 128), (1025, 48), (4097, 100), (16383, 64), (16384, 128), (20001, 130)]


@pytest.mark.parametrize("n,hidden", SIZES)
def test_gradients_and_forward(cuda, tnq_lib, n, hidden):
    torch = cuda
    from paper_2004_10892_gb300 import learned as LN

    F = LN.features()
    rng = np.random.default_rng(n + hidden)
    X = rng.random((n, F)).astype(np.float32)
    y = rng.standard_normal(n).astype(np.float32)
    p = LN.init_params(7, hidden)
    p += (0.01 * rng.standard_normal(p.size)).astype(np.float32)  # biases too
    dev = [torch.from_numpy(a).cuda() for a in (p, X, y)]
    loss, g = LN.gpu_grad(*dev, hidden)
    again_loss, again = LN.gpu_grad(*dev, hidden)
    assert torch.equal(g, again) and torch.equal(loss, again_loss)  # fixed order
    ref_loss, ref_g = omlp.loss_and_grad(p, X, y, F, hidden)
    g = g.cpu().numpy()
    assert abs(float(loss) - ref_loss) <= 1e-5 * max(1.0, ref_loss)
    assert np.linalg.norm(g - ref_g) <= 1e-5 * np.linalg.norm(ref_g)
    out = LN.gpu_forward(dev[0], dev[1], hidden).cpu().numpy()
    ref, _ = omlp.forward(p, X, F, hidden)
    assert np.max(np.abs(out - ref)) <= 1e-5 * max(1.0, np.max(np.abs(ref)))
