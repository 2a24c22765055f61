"""The warm-start network's sizes past 32-bit indices."""
import pytest

import paper_1908_07392_gb300 as V

pytestmark = pytest.mark.gpu


# a layer of 46341^2 = 2^31 + 4633 weights: outputs and gradients of its first, middle and last rows against FP64 sums
# of the same parameters (about 60 GB on the device, 9 GB on the host). A sum of 46341 products in FP32, one after the
# other: 46342 U of the sum of magnitudes at worst.
def test_a_layer_of_2_to_the_31_weights():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available() or torch.cuda.mem_get_info()[0] < 90e9:
        pytest.skip("needs a CUDA device with 90 GB free")
    c, n, U = 46341, 4, 2.0 ** -24
    net = V.WarmStartNet(in_ch=c, width=1, out_ch=c, n_layers=1, ksize=1, n=n, max_batch=1, seed=2)
    try:
        g = torch.Generator(device="cuda").manual_seed(4)
        x, t = (torch.randn(1, c, n, generator=g, device="cuda") for _ in range(2))
        p, y = net.params(), net.forward(x)
        grad, _ = net.grad(x, t)
        W, b, dW, db = p[:c * c].view(c, c), p[c * c:], grad[:c * c].view(c, c), grad[c * c:]
        x64 = x[0].double()
        for rows in (slice(0, 3), slice(c // 2, c // 2 + 3), slice(c - 3, c)):
            ref = W[rows].double() @ x64 + b[rows, None].double()
            mag = W[rows].double().abs() @ x64.abs() + b[rows, None].double().abs()
            assert ((y[0, rows].double() - ref).abs() <= (c + 1) * U * mag).all()
            dz = 2.0 * (y[0, rows].double() - t[0, rows].double()) / (c * n)
            assert ((dW[rows].double() - dz @ x64.t()).abs() <= 16 * U * (dz.abs() @ x64.abs().t())).all()
            assert ((db[rows].double() - dz.sum(1)).abs() <= 16 * U * dz.abs().sum(1)).all()
    finally:
        net.close()
