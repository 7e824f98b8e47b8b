"""Training takes the rows once and a bounded number of batches beside them."""
import numpy as np
import pytest

from paper_2004_10892_gb300 import learned

pytestmark = pytest.mark.gpu


def test_device_memory_of_training(cuda, tnq_lib):
    rows, batch, hidden = 1 << 20, 1024, 16
    rng = np.random.default_rng(0)
    X = rng.random((rows, learned.features()), dtype=np.float32)
    y = rng.random(rows, dtype=np.float32)
    learned.train(X[:batch], y[:batch], epochs=1, batch=batch, hidden=hidden)
    cuda.cuda.synchronize()
    before = cuda.cuda.memory_allocated()
    cuda.cuda.reset_peak_memory_stats()
    learned.train(X, y, epochs=2, batch=batch, hidden=hidden)
    used = cuda.cuda.max_memory_allocated() - before
    row = X[0].nbytes + 4
    # the rows, two permutations of 64-bit numbers at an epoch's turn, 64 batches, work space of one
    assert used <= rows * (row + 16) + 65 * batch * row + 4 * (batch * (5 * hidden + 4) + 16) + (4 << 20)


@pytest.mark.parametrize("rows,batch", [(66 * 32 + 5, 32), (64 * 32, 32), (100, 100), (70, 1000), (65 * 16, 16)])
def test_batches_of_every_epoch(cuda, tnq_lib, rows, batch):
    """Weights and losses of training against the same steps one call at a time: the same bits."""
    hidden = 16
    rng = np.random.default_rng(rows)
    X = rng.random((rows, learned.features()), dtype=np.float32)
    y = rng.random(rows, dtype=np.float32)
    w, hist = learned.train(X, y, epochs=2, batch=batch, lr=0.02, mu=0.9, seed=3, hidden=hidden)
    b = min(batch, rows)
    p = cuda.from_numpy(learned.init_params(3, hidden)).cuda()
    m = cuda.zeros_like(p)
    g = cuda.Generator(device="cpu").manual_seed(3)
    for e in range(2):
        perm, total = cuda.randperm(rows, generator=g), 0.0
        for i in range(0, rows - b + 1, b):
            at = perm[i:i + b].numpy()
            xb, yb = cuda.from_numpy(X[at]).cuda(), cuda.from_numpy(y[at]).cuda()
            loss, grad = learned.gpu_grad(p, xb, yb, hidden)
            tnq_lib._check(tnq_lib.lib().tnq_mlp_sgd(learned._dptr(p), learned._dptr(grad), learned._dptr(m), p.numel(),
                                                     0.02, 0.9, tnq_lib._stream_ptr(None)))
            total += float(loss)
        assert hist[e] == total / (rows // b)
    assert np.array_equal(w, p.cpu().numpy())
