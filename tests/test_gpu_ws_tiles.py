"""The warm-start network's convolution and weight-gradient tiles at their edges: ragged lengths, channel
counts around the tile sizes (2, 8, 16, 64 output channels, odd input channels), every kind of kernel size, small
and large launches, against the FP64 oracle with rounding bounds of FP32 sums."""
import numpy as np
import pytest

import paper_1908_07392_gb300 as V
from oracle import ws_oracle as WO

pytestmark = pytest.mark.gpu

U = 2.0 ** -24


def net_and_data(cin, width, cout, layers, K, n, B, seed):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    rng = np.random.default_rng(seed)
    net = V.WarmStartNet(in_ch=cin, width=width, out_ch=cout, n_layers=layers, ksize=K, n=n, max_batch=B, seed=seed)
    x = rng.standard_normal((B, cin, n)).astype(np.float32)
    t = rng.standard_normal((B, cout, n)).astype(np.float32)
    p = net.params().cpu().numpy().astype(np.float64)
    return net, x, t, p


# one layer: every output is a sum of cin K products (and the bias) of FP32 numbers, so its error is below
# (cin K + 1) U sum |w| |x|; a weight gradient sums B n products, its dz carries 4 roundings
@pytest.mark.parametrize("cin,cout,K,n,B", [(1, 1, 1, 5, 1), (3, 2, 3, 130, 2), (10, 5, 5, 33, 3), (9, 64, 9, 257, 1),
                                            (7, 70, 7, 61, 2), (65, 17, 11, 128, 2), (16, 48, 13, 200, 2),
                                            (20, 64, 15, 520, 1), (64, 64, 9, 1000, 40), (8, 66, 3, 4096, 12)])
def test_one_layer(cin, cout, K, n, B):
    import torch
    net, x, t, p = net_and_data(cin, 4, cout, 1, K, n, B, cin + K)
    try:
        y = net.forward(torch.tensor(x, device="cuda")).cpu().numpy().astype(np.float64)
        g, loss = net.grad(torch.tensor(x, device="cuda"), torch.tensor(t, device="cuda"))
        g = g.cpu().numpy().astype(np.float64)
    finally:
        net.close()
    W, b = p[:cout * cin * K].reshape(cout, cin, K), p[cout * cin * K:]
    x64 = x.astype(np.float64)
    cols = np.stack([np.roll(x64, K // 2 - k, axis=2) for k in range(K)], axis=2)  # [B][cin][K][n]
    ref = np.einsum("ock,bckx->box", W, cols) + b[None, :, None]
    mag = np.einsum("ock,bckx->box", np.abs(W), np.abs(cols)) + np.abs(b)[None, :, None]
    assert (np.abs(y - ref) <= (cin * K + 1) * U * mag).all()
    dz = 2.0 * (ref - t) / ref.size
    assert loss == pytest.approx(((ref - t) ** 2).mean(), rel=1e-5)
    err_dz = 2.0 / ref.size * (cin * K + 1) * U * mag + 4 * U * np.abs(dz)
    gw = np.einsum("box,bckx->ock", dz, cols)
    bound = np.einsum("box,bckx->ock", (B * n + 320) * U * np.abs(dz) + err_dz, np.abs(cols))
    assert (np.abs(g[:gw.size].reshape(gw.shape) - gw) <= bound).all()
    assert (np.abs(g[gw.size:] - dz.sum((0, 2))) <= ((B * n + 320) * U * np.abs(dz) + err_dz).sum((0, 2))).all()


# three layers: the transposed convolution with the fused mask; norms of the difference, FP32 sums of up to
# 576 terms twice over (about 600 U sqrt(layers) at worst)
@pytest.mark.parametrize("cin,width,K,n,B", [(5, 6, 3, 50, 2), (10, 64, 9, 300, 2), (11, 33, 5, 129, 16),
                                             (10, 64, 9, 1024, 40)])
def test_three_layers(cin, width, K, n, B):
    import torch
    net, x, t, p = net_and_data(cin, width, 2, 3, K, n, B, width + K)
    try:
        y = net.forward(torch.tensor(x, device="cuda")).cpu().numpy()
        g, _ = net.grad(torch.tensor(x, device="cuda"), torch.tensor(t, device="cuda"))
        g2, _ = net.grad(torch.tensor(x, device="cuda"), torch.tensor(t, device="cuda"))
        assert torch.equal(g, g2)
        g = g.cpu().numpy()
    finally:
        net.close()
    chans = [cin, width, width, 2]
    _, go = WO.loss_and_grad(p, chans, K, x.astype(np.float64), t.astype(np.float64))
    assert np.linalg.norm(g - go) <= 6e-5 * np.linalg.norm(go)
    assert np.isfinite(y).all()
