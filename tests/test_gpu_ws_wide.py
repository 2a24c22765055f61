"""The warm-start network's wide layers: sizes past 32-bit indices, and the rounding of the weight gradient's sums."""
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


# With zero weights and as many outputs as a power of two, dz = -2 t / m exactly, so the gradient is the sum over
# the positions alone; products of one sign make its rounding plain. A chunk of 64 positions is a segment of its own here:
# at most 8 + 8 roundings of a term and 2 of the compensated sum over segments. Independent roundings (U / sqrt 3 of the
# partial sum each): 8 blocks of 8 leave 121 units of a term in the 64 of a chunk, 1.9 / sqrt(chunks) U / sqrt 3 of the sum,
# and rounding the result 1 more: below 1.2 U for any number of chunks.
@pytest.mark.parametrize("cin,cout,K,n,B", [(512, 512, 15, 512, 4), (320, 256, 9, 256, 2), (64, 64, 9, 1024, 4),
                                            (130, 64, 3, 64, 2)])
def test_rounding_of_the_weight_gradient(cin, cout, K, n, B):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    U = 2.0 ** -24
    net = V.WarmStartNet(in_ch=cin, width=1, out_ch=cout, n_layers=1, ksize=K, n=n, max_batch=B, seed=2)
    try:
        net.set_params(torch.zeros(net.n_params, device="cuda"))
        gen = torch.Generator(device="cuda").manual_seed(7)
        x = 1 + torch.rand(B, cin, n, generator=gen, device="cuda")
        t = -1 - torch.rand(B, cout, n, generator=gen, device="cuda")
        g, _ = net.grad(x, t)
    finally:
        net.close()
    dz, x64 = -2.0 * t.double() / t.numel(), x.double()
    for k in range(K):
        ref = torch.einsum("box,bcx->oc", dz, torch.roll(x64, K // 2 - k, dims=2))
        err = (g[:cout * cin * K].view(cout, cin, K)[:, :, k].double() - ref) / ref
        assert float(err.abs().max()) <= 18 * U
        assert float(err.square().mean().sqrt()) <= 1.2 * U
    err = (g[cout * cin * K:].double() - dz.sum((0, 2))) / dz.sum((0, 2))
    assert float(err.abs().max()) <= 18 * U
