"""The network's products at the edges of their tiles (128 rows, 32 columns, K blocks of 128 in steps of 16)."""
import os

import numpy as np
import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def S():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1811_10270_gb300 as pkg
    if not os.path.exists(pkg.LIB_PATH):
        from paper_1811_10270_gb300 import build
        build.build()
    pkg.lib()
    return pkg


def half(a):
    """Rounded to bfloat16, as the products read it, in 64 bits."""
    return torch.as_tensor(np.asarray(a)).float().bfloat16().double().numpy()


def close(got, a, b, add=0.0):
    """got against a @ b in 64 bits: each 16 terms of K enter the FP32 accumulator with an error of at most
    2^-22 of sum |a| |b| (one rounding or truncation of the partial sum and one of the 16 products)."""
    ref = a @ b + add
    bound = (a.shape[1] / 16 + 2) * 2.0**-22 * (np.abs(a) @ np.abs(b) + np.abs(add))
    assert np.all(np.abs(got - ref) <= bound)


@pytest.mark.parametrize("widths,batch", [([1, 5, 1], 5), ([129, 33, 32], 16), ([128, 31, 65], 17),
                                          ([257, 128, 130], 128), ([657, 129, 66], 131)])
def test_products_at_tile_edges(S, widths, batch):
    rng = np.random.default_rng(batch)
    Ws = [(rng.uniform(-1, 1, (b, a)) / np.sqrt(a)).astype(np.float32) for a, b in zip(widths, widths[1:])]
    bs = [rng.standard_normal(b).astype(np.float32) for b in widths[1:]]
    x = rng.standard_normal((batch, widths[0])).astype(np.float32)
    t = rng.standard_normal((batch, widths[2])).astype(np.float32)
    X, Y = torch.tensor(x, device="cuda"), torch.empty(batch, widths[2], device="cuda")
    # one layer: the forward product by itself
    for l, inp in ((0, x), (1, rng.standard_normal((batch, widths[1])).astype(np.float32))):
        one = S.MLP(widths[l:l + 2], max_batch=batch)
        one.set_layer(0, Ws[l], bs[l])
        y = torch.empty(batch, widths[l + 1], device="cuda")
        one.forward(torch.tensor(inp, device="cuda"), y)
        close(y.cpu().numpy(), half(inp), half(Ws[l]).T, bs[l].astype(np.float64))
        one.close()
    net = S.MLP(widths, max_batch=batch)
    for l in range(2):
        net.set_layer(l, Ws[l], bs[l])
    net.train_step(X, torch.tensor(t, device="cuda"), 0.0, update=False)
    net.forward(X, Y)
    h = np.tanh(half(x) @ half(Ws[0]).T + bs[0])
    d = (Y.cpu().numpy() - t) * np.float32(1.0 / batch)
    _, _, g1, b1 = net.get_layer(1)
    _, _, g0, b0 = net.get_layer(0)
    # operands of these are rounded from FP32 values that are known to FP32 only: a rounding to bfloat16 that falls
    # the other way is 2^-8 of its element, and few do
    rel = lambda a, b: np.linalg.norm(a - b) / np.linalg.norm(b)
    assert rel(g1, half(d).T @ half(h)) < 2.0**-8
    dn = (half(d) @ half(Ws[1])) * (1 - h * h)
    assert rel(g0, half(dn).T @ half(x)) < 2.0**-8
    np.testing.assert_allclose(b1, d.astype(np.float64).sum(0), rtol=0, atol=batch * 2.0**-24 * np.abs(d).sum(0).max())
    assert rel(b0, dn.sum(0)) < 2.0**-8
    net.close()
