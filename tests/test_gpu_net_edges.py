"""The network's GEMMs at the edges of their tiles and of the cluster split of the
inner dimension (one chunk of 64 per CTA up to 8, then several chunks per CTA, ranks
without chunks): forward, loss and gradient against the FP64 oracle.  Bars: FP32 sums
of n terms, a few ulp times sqrt(n) of the largest entry (1e-5 forward, 1e-4 gradient,
those of the network's oracle test)."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("sizes,batch", [([1, 1, 1], 1), ([63, 33, 65], 31), ([65, 32, 31], 33), ([64, 5], 64),
                                         ([513, 40, 97], 2), ([577, 65, 600], 100), ([1300, 17, 9], 257)])
def test_gemm_edges(sizes, batch):
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
    # an Adam step without a loss request takes the same gradient
    a, b = Net(sizes, batch, p), Net(sizes, batch, p)
    a.adam_step(Xd, Td, batch, 1e-3, want_loss=True)
    b.adam_step(Xd, Td, batch, 1e-3)
    assert np.array_equal(a.params(), b.params())
    for n in (net, a, b):
        n.close()
