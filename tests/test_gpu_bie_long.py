"""Boundary solves that leave the one-launch Arnoldi step: subspaces past its 64 columns, with and without an augmentation
direction, and more unknowns than its 32768; and the operator's fixed-point entries against the kernel's closed form."""
import numpy as np
import pytest

import paper_1908_07392_gb300 as V

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    V.load_library()


# a tolerance that the residual's estimate (about 1e-45 after 70 steps) does not reach; the true residual ends at rounding
# level, and the solution is that of the short solve (residual 2e-11, condition below 50)
@pytest.mark.parametrize("panels", [4, 37, 300])
@pytest.mark.parametrize("aug", [False, True])
def test_subspaces_past_the_one_launch_limit(panels, aug):
    import torch
    b = V.BIE(25.0, phase=0.1, n_panels=panels, max_krylov=80)
    try:
        n, th = 2 * b.N, b.nodes[6]
        g = torch.stack([torch.cos(3 * th) + b.nodes[0], torch.sin(2 * th) * b.nodes[1]], 1).reshape(-1).contiguous()
        d = torch.from_numpy(np.random.default_rng(panels).standard_normal(n)).cuda() if aug else None
        mu, it, rr = b.solve(g, tol=1e-11)
        assert rr <= 2e-11 and 0 < it < 64
        long_mu, it, rr = b.solve(g, tol=1e-300, max_iter=70, aug=d)
        assert it == 70 and rr <= 1e-14
        assert torch.linalg.norm(long_mu - mu) <= 1e-9 * torch.linalg.norm(mu)
    finally:
        b.close()


# 32768 unknowns (one launch a step) and 32800 (separate kernels): as many steps, and inside the star the velocity of the
# stokeslets outside that the boundary values are taken from
def test_more_unknowns_than_the_one_launch_limit():
    import torch
    if torch.cuda.mem_get_info()[0] < 30e9:
        pytest.skip("needs 30 GB of device memory")
    rng = np.random.default_rng(4)
    th, r = rng.uniform(0, 2 * np.pi, 3), rng.uniform(1.6, 2.0, 3)
    src = torch.from_numpy(np.stack([r * np.cos(th), r * np.sin(th)], axis=1)).cuda()
    f = torch.from_numpy(rng.uniform(-1, 1, (3, 2))).cuda()
    th, r = rng.uniform(0, 2 * np.pi, 40), 0.4 * np.sqrt(rng.uniform(0, 1, 40))
    xy = torch.from_numpy(np.stack([r * np.cos(th), r * np.sin(th)])).cuda()
    exact = V.bie_stokeslets(6.0, src, f, xy)
    steps = []
    for panels in (1024, 1025):
        b = V.BIE(6.0, phase=0.2, n_panels=panels, max_krylov=50)
        try:
            g = V.bie_stokeslets(6.0, src, f, b.nodes[:2].contiguous()).t().reshape(-1).contiguous()
            mu, it, rr = b.solve(g, tol=1e-12)
            assert rr <= 2e-12
            assert float((b.eval(mu, xy) - exact).abs().max()) <= 1e-9 * float(exact.abs().max())
            steps.append(it)
        finally:
            b.close()
    assert abs(steps[0] - steps[1]) <= 1


# entries of columns far from their panel: the kernel times the weight and the rank-one term, from torch's Bessel
# functions (about 1e-15 of the terms each) and rounded to 2^-63 of the row's largest entry; whole rows come from
# applying the unit vectors
@pytest.mark.parametrize("alpha", [5.0, 60.0])
def test_entries_of_the_operator(alpha):
    import torch
    b = V.BIE(alpha, phase=0.3, n_panels=8, max_krylov=1)
    try:
        N = b.N
        A = torch.stack([b.apply(e) for e in torch.eye(2 * N, dtype=torch.float64, device="cuda")], dim=1)
        x, y, nx, ny, w = b.nodes[:5]
        R = torch.stack([x[:, None] - x, y[:, None] - y])
        r2 = (R * R).sum(0) + torch.eye(N, dtype=torch.float64, device="cuda")
        z = alpha * r2.sqrt()
        k0, k1 = torch.special.modified_bessel_k0(z), torch.special.modified_bessel_k1(z)
        T = [-(2 * z ** 2 * k0 + (z ** 2 + 4) * z * k1 - 4) / (2 * np.pi * z ** 4) * alpha ** 2,
             (4 * z ** 2 * k0 + (z ** 2 + 8) * z * k1 - 8) / (np.pi * z ** 6) * alpha ** 4,
             (z * k1 - 1) / (2 * np.pi * z ** 2) * alpha ** 2]
        lost = [(2 * z ** 2 * k0 + (z ** 2 + 4) * z * k1 + 4) / (2 * np.pi * z ** 4) * alpha ** 2,
                (4 * z ** 2 * k0 + (z ** 2 + 8) * z * k1 + 8) / (np.pi * z ** 6) * alpha ** 4,
                (z * k1 + 1) / (2 * np.pi * z ** 2) * alpha ** 2]  # sums of magnitudes before cancellation
        nn = torch.stack([nx, ny])
        rn = (R * nn[:, None]).sum(0)
        p = torch.arange(N, device="cuda") // 16
        gap = (p[:, None] - p).abs()
        far = torch.minimum(gap, 8 - gap) >= 2
        length = w.sum()
        for i in range(2):
            for j in range(2):
                parts = [nn[i] * R[j] + R[i] * nn[j] + (rn if i == j else 0.0), R[i] * R[j] * rn, R[i] * nn[j]]
                wall = nn[i][:, None] * nn[j] * w / length
                ref = -sum(t * q for t, q in zip(T, parts)) * w + wall
                mag = sum(m * q.abs() for m, q in zip(lost, parts)) * w + wall.abs()
                rows = A[i::2].abs().amax(1, keepdim=True)
                got = A[i::2, j::2]
                assert ((got - ref).abs() <= 1e-14 * mag + 2.0 ** -62 * rows)[far].all()
    finally:
        b.close()
