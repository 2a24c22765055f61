"""The warm-start network's training step keeps every form of the weights in step: after it, forward passes and
gradients are those of a new network with the same parameters, bit for bit."""
import pytest

import paper_1908_07392_gb300 as V

pytestmark = pytest.mark.gpu


# one to five layers, channel counts that are padded to 4 and that are not, one chunk of positions (whose gradient is
# written at once) and more
@pytest.mark.parametrize("cin,width,cout,L,K,n,B", [(1, 1, 1, 1, 1, 5, 1), (1, 4, 1, 2, 1, 16, 1), (3, 7, 2, 3, 3, 64, 1),
                                                    (10, 66, 5, 4, 5, 65, 1), (10, 16, 2, 5, 9, 200, 3)])
def test_weights_after_training_steps(cin, width, cout, L, K, n, B):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    shape = dict(in_ch=cin, width=width, out_ch=cout, n_layers=L, ksize=K, n=n, max_batch=B)
    a, b = V.WarmStartNet(seed=1, **shape), V.WarmStartNet(seed=2, **shape)
    try:
        gen = torch.Generator(device="cuda").manual_seed(3)
        x, t = (torch.randn(B, c, n, generator=gen, device="cuda") for c in (cin, cout))
        before = a.params()
        losses = [a.train_step(x, t, 1e-2) for _ in range(3)]
        p = a.params()
        assert not torch.equal(p, before) and losses[2] < losses[0]
        b.set_params(p)
        assert torch.equal(a.forward(x), b.forward(x))
        (ga, la), (gb, lb) = a.grad(x, t), b.grad(x, t)
        assert torch.equal(ga, gb) and la == lb
        # the gradient against autograd of the same network in FP64
        q, h, at = p.double().requires_grad_(True), x.double(), 0
        chans = [cin] + [width] * (L - 1) + [cout]
        for l in range(L):
            m = chans[l + 1] * chans[l] * K
            W, bias = q[at:at + m].view(chans[l + 1], chans[l], K), q[at + m:at + m + chans[l + 1]]
            at += m + chans[l + 1]
            h = sum(torch.einsum("oc,bcx->box", W[:, :, k], torch.roll(h, K // 2 - k, dims=2)) for k in range(K))
            h = h + bias[None, :, None]
            h = torch.relu(h) if l < L - 1 else h
        ((h - t.double()) ** 2).mean().backward()
        assert torch.linalg.norm(ga.double() - q.grad) <= 6e-5 * torch.linalg.norm(q.grad)
    finally:
        a.close(); b.close()
