"""The network's 64 x 64 tiles (products of 128 of them and more that are not half empty):
ragged edges, inner dimensions around the chunks of 64, either side of the rule, against
the FP64 oracle.  Bars: those of the network's other GEMM tests (1e-5 forward, 1e-4 of
the largest gradient)."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu


# tiles of 64: 8 x 16 = 128 (just there), 8 x 15 (not); ragged by one row or column; inner
# dimensions 1, 63, 64, 65, 129, 640; weight gradients of 128 tiles and more
@pytest.mark.parametrize("sizes,batch", [([64, 1024], 512), ([64, 960], 512), ([1, 1025], 513), ([63, 1023], 511),
                                         ([65, 1100, 3], 600), ([129, 2000, 300], 300), ([640, 1030, 640], 577),
                                         ([40, 32, 4100], 130), ([33, 32], 9000)])
def test_wide_products(sizes, batch):
    from oracle import mlp
    from paper_2211_13893_gb300 import Net
    rng = np.random.default_rng(3)
    p = (rng.standard_normal(mlp.param_count(sizes)) / np.sqrt(max(sizes))).astype(np.float32)
    X = rng.standard_normal((batch, sizes[0])).astype(np.float32)
    T = rng.standard_normal((batch, sizes[-1])).astype(np.float32)
    net = Net(sizes, batch, p)
    Xd, Td = torch.tensor(X, device="cuda"), torch.tensor(T, device="cuda")
    Y = torch.empty((batch, sizes[-1]), dtype=torch.float32, device="cuda")
    net.forward(Xd, Y, batch)
    ref, _ = mlp.forward(p.astype(np.float64), sizes, X.astype(np.float64))
    assert np.max(np.abs(Y.cpu().numpy() - ref)) <= 1e-5 * np.max(np.abs(ref))
    loss, g = net.gradient(Xd, Td, batch)
    loss_ref, g_ref = mlp.backward(p.astype(np.float64), sizes, X.astype(np.float64), T.astype(np.float64))
    assert loss == pytest.approx(loss_ref, rel=1e-5)
    assert np.max(np.abs(g - g_ref)) <= 1e-4 * np.max(np.abs(g_ref))
    net.close()
