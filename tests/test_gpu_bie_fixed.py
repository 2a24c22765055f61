"""The boundary operator in fixed point, the one-launch Arnoldi step and the far evaluation at their edges:
segments of the vector, row counts that do not divide among the SMs, subspaces past the one-launch limit, the
augmented solve, and targets on both sides of the far rule."""
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


# A e_j returns the column to FP64, so A x of a vector with a few components is known in extended precision. 31 to 260
# panels: one segment (n <= 8192) and two. Each term is rounded to 2^-53 of itself twice, the sum once.
@pytest.mark.parametrize("panels", [4, 31, 256, 257, 260])
def test_apply_is_the_sum_of_its_columns(panels):
    import torch
    b = V.BIE(40.0, phase=0.3, n_panels=panels, max_krylov=1)
    try:
        n = 2 * b.N
        rng = np.random.default_rng(panels)
        at = np.unique(np.concatenate([[0, 1, n - 1, n // 2, min(n - 1, 8191), min(n - 1, 8192)], rng.integers(0, n, 10)]))
        val = rng.standard_normal(at.size) * 10.0 ** rng.uniform(-9, 0, at.size)
        x, ref, mag = np.zeros(n), np.zeros(n, np.longdouble), np.zeros(n)
        for j, v in zip(at, val):
            e = torch.zeros(n, dtype=torch.float64, device="cuda")
            e[int(j)] = 1.0
            col = b.apply(e).cpu().numpy()
            x[j] = v
            ref += col.astype(np.longdouble) * v
            mag += np.abs(col * v)
        y = b.apply(torch.from_numpy(x).cuda()).cpu().numpy()
        assert (np.abs(y - ref.astype(np.float64)) <= 4 * 2.0 ** -53 * mag + 1e-300).all()
        x[n // 3] = np.nan
        assert np.isnan(b.apply(torch.from_numpy(x).cuda()).cpu().numpy()).all()
        assert not b.apply(torch.zeros(n, dtype=torch.float64, device="cuda")).any()
    finally:
        b.close()


# a tolerance that is not reached runs the subspace past the one-launch limit of 64 columns (and of 32768 unknowns never);
# the residual ends at rounding level, and the augmented solve agrees
@pytest.mark.parametrize("panels", [4, 37, 300])
def test_long_and_augmented_solves(panels):
    import torch
    b = V.BIE(25.0, phase=0.1, n_panels=panels, max_krylov=80)
    try:
        n = 2 * b.N
        th = b.nodes[6]
        g = torch.stack([torch.cos(3 * th) + b.nodes[0], torch.sin(2 * th) * b.nodes[1]], 1).reshape(-1).contiguous()
        mu, it, rr = b.solve(g, tol=1e-11)
        assert rr <= 2e-11 and 0 < it < 64
        long_mu, it, rr = b.solve(g, tol=1e-30, max_iter=70)
        assert rr <= 1e-14
        assert torch.linalg.norm(long_mu - mu) <= 1e-9 * torch.linalg.norm(mu)
        d = torch.from_numpy(np.random.default_rng(panels).standard_normal(n)).cuda()
        aug, _, rr = b.solve(g, tol=1e-11, aug=d)
        assert rr <= 2e-11 and torch.linalg.norm(aug - mu) <= 1e-9 * torch.linalg.norm(mu)
        assert torch.equal(b.solve(g, tol=1e-11)[0], mu)
    finally:
        b.close()


# alpha r below the far rule (50), on both sides of it and beyond it, against the closed forms in FP64 by torch; an
# odd number of targets. Both sums carry about 1e-15 of the sum of their terms' magnitudes.
@pytest.mark.parametrize("alpha", [20.0, 60.0, 250.0])
def test_evaluation_on_both_sides_of_the_far_rule(alpha):
    import torch
    b = V.BIE(alpha, phase=0.2, n_panels=40, max_krylov=1)
    try:
        rng = np.random.default_rng(5)
        r, th = 0.55 * np.sqrt(rng.uniform(0, 1, 201)), rng.uniform(0, 2 * np.pi, 201)
        xy = torch.from_numpy(np.stack([r * np.cos(th), r * np.sin(th)])).cuda()
        mu = torch.from_numpy(rng.standard_normal(2 * b.N)).cuda()
        u = b.eval(mu, xy)
        x, y, nx, ny, w = b.nodes[:5]
        m = mu.view(-1, 2).t() * w
        R = torch.stack([xy[0][:, None] - x, xy[1][:, None] - y])
        r2 = (R * R).sum(0)
        z = alpha * r2.sqrt()
        k0, k1 = torch.special.modified_bessel_k0(z), torch.special.modified_bessel_k1(z)
        T1 = -(2 * z ** 2 * k0 + (z ** 2 + 4) * z * k1 - 4) / (2 * np.pi * z ** 4) * alpha ** 2
        T2 = (4 * z ** 2 * k0 + (z ** 2 + 8) * z * k1 - 8) / (np.pi * z ** 6) * alpha ** 4
        T3 = (z * k1 - 1) / (2 * np.pi * z ** 2) * alpha ** 2
        nn = torch.stack([nx, ny])
        rn, rm, nm = (R * nn[:, None]).sum(0), (R * m[:, None]).sum(0), (nn * m).sum(0)
        for a in range(2):
            t = -T1 * (nn[a] * rm + R[a] * nm + m[a] * rn) - T2 * R[a] * rm * rn - T3 * R[a] * nm
            assert (torch.abs(u[a] - t.sum(1)) <= 2e-14 * t.abs().sum(1)).all()
    finally:
        b.close()
