"""Rounding of the entry model's hidden gradient: no larger than that of 32 strided chains
and a tree over the cells, whatever the batch size and the number of cells."""
import numpy as np
import pytest

from helpers import dev
from oracle import mlp

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def nhq():
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA device")
    from paper_2203_13601_gb300 import build as B

    B.build()
    import paper_2203_13601_gb300 as m

    m.load_library()
    return m


def _chains_and_tree(dt, w2):
    """sum_o dt[o] w2[h][o] in f32: lane l adds the cells l, l + 32, ... with one rounding
    per multiply-add, then the lanes are added pairwise."""
    E = dt.size
    pad = -E % 32
    a = np.pad(dt, (0, pad)).reshape(-1, 32).astype(np.float64)
    b = np.pad(w2, ((0, 0), (0, pad))).reshape(w2.shape[0], -1, 32).astype(np.float64)
    acc = np.zeros((w2.shape[0], 32), np.float32)
    for i in range(a.shape[0]):
        acc = (acc.astype(np.float64) + a[i] * b[:, i]).astype(np.float32)
    while acc.shape[1] > 1:
        half = acc.shape[1] // 2
        acc = acc[:, :half] + acc[:, half:]
    return acc[:, 0].astype(np.float64)


# One sample of the batch counts (the others carry no cell), so that the gradients of b2 and
# b1 are that sample's dT and dZ themselves.  Over 8 samples x 64 units the root mean squares
# of equally large errors differ by about 1 / sqrt(2 * 512) = 3 % each; 15 % is allowed.
@pytest.mark.parametrize("n,E", [(1, 64), (64, 256), (256, 4096), (129, 1000), (1024, 64),
                                 (2048, 256), (4096, 64), (4096, 1000), (3000, 4096)])
def test_hidden_gradient_rounds_no_more_than_lane_sums(nhq, n, E):
    d = 16
    rng = np.random.default_rng(n + E)
    p = (rng.standard_normal(mlp.entry_size(d, E)) * 0.2).astype(np.float32)
    p[0] = 0.3
    p[1 + 64 * d:65 + 64 * d] = 2.0  # every hidden unit is active
    w2 = p[65 + 64 * d:65 + 64 * (d + E)].reshape(64, E)
    Q = (rng.standard_normal((n, d)) * 0.1).astype(np.float32)
    P, X = dev(p), dev(Q)
    grad = torch.empty(p.size, dtype=torch.float32, device="cuda:0")
    loss = torch.empty(1, dtype=torch.float32, device="cuda:0")
    ours, lanes = [], []
    for t in range(8):
        y = np.full(n, -1, np.int32)
        y[(t * n) // 8] = rng.integers(0, E)
        nhq.nhq_entry_grad(P, E, X, dev(y), grad, loss)
        g = grad.cpu().numpy()
        dt, dz = g[65 + 64 * (d + E):], g[1 + 64 * d:65 + 64 * d].astype(np.float64)
        want = w2.astype(np.float64) @ dt.astype(np.float64)
        ours.append(dz - want)
        lanes.append(_chains_and_tree(dt, w2) - want)
        p_scale = np.abs(want).max()
        assert np.allclose(dz, want, rtol=0, atol=1e-5 * p_scale)
        if n == 1:
            X = dev((rng.standard_normal((n, d)) * 0.1).astype(np.float32))
    rms = [float(np.sqrt(np.mean(np.square(e)))) for e in (ours, lanes)]
    assert rms[0] <= 1.15 * rms[1], rms


# the kernels for few samples and their limits (128 samples, 2^18 outputs), and two chunks of
# a batch whose second one is small (2,560 + 40 samples) or not (2,560 + 200)
@pytest.mark.parametrize("d,E,n", [(3, 5, 2), (40, 300, 128), (40, 300, 129), (16, 4096, 64),
                                   (16, 4096, 65), (16, 4096, 2600), (16, 4096, 2760)])
def test_gradient_of_few_samples_and_of_several_chunks(nhq, d, E, n):
    rng = np.random.default_rng(d + E + n)
    p = (rng.standard_normal(mlp.entry_size(d, E)) * 0.2).astype(np.float32)
    p[0] = 0.5 / np.sqrt(d)
    Q = rng.standard_normal((n, d)).astype(np.float32)
    y = rng.integers(0, E, n).astype(np.int32)
    grad = torch.full((p.size,), float("nan"), dtype=torch.float32, device="cuda:0")
    loss = torch.full((1,), float("nan"), dtype=torch.float32, device="cuda:0")
    nhq.nhq_entry_grad(dev(p), E, dev(Q), dev(y), grad, loss)
    torch.cuda.synchronize()
    lw, gw = mlp.entry_loss_and_grad(p.astype(np.float64), Q, y, d, E)
    # f32 sums of at most 2,760 terms: relative 1e-4 of each sum's largest terms
    assert abs(loss.item() - lw) <= 1e-4 * abs(lw)
    assert np.allclose(grad.cpu().numpy(), gw, rtol=1e-3, atol=1e-5 * np.abs(gw).max())
