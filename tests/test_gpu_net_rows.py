"""Networks with more rows or columns than 32 times a grid's second dimension: a batch of
2,200,000 and a layer of as many units, against the FP64 oracle on samples of the rows
(bars of the network's other GEMM tests: 1e-5 forward, 1e-4 of the largest gradient)."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu

BIG = 2_200_000


def _setup(sizes, batch):
    from oracle import mlp
    from paper_2211_13893_gb300 import Net
    rng = np.random.default_rng(3)
    p = (rng.standard_normal(mlp.param_count(sizes)) / 2.0).astype(np.float32)
    X = rng.standard_normal((batch, sizes[0])).astype(np.float32)
    net = Net(sizes, batch, p)
    return mlp, p, X, net, torch.tensor(X, device="cuda")


def test_long_batch():
    sizes = [3, 5, 2]
    mlp, p, X, net, Xd = _setup(sizes, BIG)
    Y = torch.zeros((BIG, sizes[-1]), dtype=torch.float32, device="cuda")
    net.forward(Xd, Y, BIG)
    pick = np.concatenate([np.arange(5), [32 * 65535 - 1, 32 * 65535, 32 * 65535 + 1], np.arange(BIG - 40, BIG)])
    ref, _ = mlp.forward(p.astype(np.float64), sizes, X[pick].astype(np.float64))
    assert np.max(np.abs(Y[torch.tensor(pick, device="cuda")].cpu().numpy() - ref)) <= 1e-5 * np.max(np.abs(ref))
    T = torch.ones_like(Y)
    loss, g = net.gradient(Xd, T, BIG)
    loss_ref, g_ref = mlp.backward(p.astype(np.float64), sizes, X.astype(np.float64), np.ones((BIG, sizes[-1])))
    assert loss == pytest.approx(loss_ref, rel=1e-5)
    assert np.max(np.abs(g - g_ref)) <= 1e-4 * np.max(np.abs(g_ref))
    net.close()


def test_wide_layer():
    sizes = [2, BIG]
    mlp, p, X, net, Xd = _setup(sizes, 3)
    Y = torch.zeros((3, BIG), dtype=torch.float32, device="cuda")
    net.forward(Xd, Y, 3)
    ref, _ = mlp.forward(p.astype(np.float64), sizes, X.astype(np.float64))
    assert np.max(np.abs(Y.cpu().numpy() - ref)) <= 1e-5 * np.max(np.abs(ref))
    T = torch.ones_like(Y)
    _, g = net.gradient(Xd, T, 3)
    _, g_ref = mlp.backward(p.astype(np.float64), sizes, X.astype(np.float64), np.ones((3, BIG)))
    assert np.max(np.abs(g - g_ref)) <= 1e-4 * np.max(np.abs(g_ref))
    net.close()
