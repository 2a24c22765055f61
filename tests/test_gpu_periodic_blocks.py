"""The periodic solution's block floating point: every transform length (last stages of radix 8, 4 and 2,
several rows per block, one or two derivatives per thread group) on white noise, which fills the Nyquist
row and column, against the numpy oracle; exact scaling by powers of two; zeros and non-finite forces."""
import numpy as np
import pytest

import paper_1908_07392_gb300 as V
from oracle import periodic_oracle as PO

pytestmark = pytest.mark.gpu

# Each of the four passes rounds to about 2^-57 of a row's largest value and twice to FP64: a few 1e-16 of
# the largest output; numpy's transforms add about as much. 1e-13 leaves two orders for the maximum over
# the points and for u dominated by its lowest modes.
TOL = 1e-13


def solve(F, alpha, L=3.0):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    P = V.PeriodicStokes(alpha, F.shape[-1], L)
    try:
        u, g = P(torch.from_numpy(np.ascontiguousarray(F)).cuda())
        torch.cuda.synchronize()
        return u.cpu().numpy(), g.cpu().numpy()
    finally:
        P.close()


@pytest.mark.parametrize("n,alpha", [(32, 3.0), (64, 30.0), (128, 3.0), (256, 316.0), (512, 3.0), (1024, 30.0),
                                     (2048, 316.0), (4096, 30.0)])
def test_white_noise(n, alpha):
    F = np.random.default_rng(n).standard_normal((2, n, n))
    F[0] += 0.5
    u, g = solve(F, alpha)
    uo, go = PO.periodic_stokes(alpha, 3.0, F)
    for a in range(2):
        assert np.abs(u[a] - uo[a]).max() <= TOL * np.abs(uo[a]).max()
        for m in range(2):
            assert np.abs(g[a, m] - go[a, m]).max() <= TOL * np.abs(go[a, m]).max()


@pytest.mark.parametrize("n", [32, 256, 1024])
def test_powers_of_two_scale_exactly_and_zero_is_zero(n):
    F = np.random.default_rng(n).standard_normal((2, n, n))
    F[:, n // 3] = 0.0     # a row of zeros among the others
    F[1, :, 5] *= 1e-30    # elements far below the row's unit
    u, g = solve(F, 10.0)
    for s in (2.0 ** 300, 2.0 ** -300):
        us, gs = solve(F * s, 10.0)
        assert np.array_equal(us, u * s) and np.array_equal(gs, g * s)
    u, g = solve(np.zeros((2, n, n)), 10.0)
    assert not u.any() and not g.any()


@pytest.mark.parametrize("bad", [np.inf, -np.inf, np.nan])
def test_non_finite_force_gives_nan_everywhere(bad):
    F = np.random.default_rng(7).standard_normal((2, 64, 64))
    F[1, 3, 60] = bad
    u, g = solve(F, 10.0)
    assert np.isnan(u).all() and np.isnan(g).all()
