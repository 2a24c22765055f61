"""The periodic solution over the whole range of alpha: the multiplier reaches 1 / alpha^2 without overflow on the way."""
import numpy as np
import pytest

import paper_1908_07392_gb300 as V
from oracle import periodic_oracle as PO

pytestmark = pytest.mark.gpu


# the mean of the force alone becomes huge for small alpha; the gradient does not see it. 1e-13 as for the other
# solutions; the largest mean, 6.5e4 over alpha^2, is finite from 1e-151 on
@pytest.mark.parametrize("n", [32, 512])
@pytest.mark.parametrize("alpha", [1e-151, 1e-148, 1e-140, 1e-60, 1e-3, 0.7, 1.0, 1e60, 1e140])
def test_any_alpha(n, alpha):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    F = np.random.default_rng(n).standard_normal((2, n, n)) + 0.25
    P = V.PeriodicStokes(alpha, n, 3.0)
    try:
        u, g = (t.cpu().numpy() for t in P(torch.from_numpy(F).cuda()))
    finally:
        P.close()
    uo, go = PO.periodic_stokes(alpha, 3.0, F)
    assert np.isfinite(uo).all() and np.isfinite(go).all()
    for a in range(2):
        assert np.abs(u[a] - uo[a]).max() <= 1e-13 * np.abs(uo[a]).max()
        for m in range(2):
            assert np.abs(g[a, m] - go[a, m]).max() <= 1e-13 * np.abs(go[a, m]).max()
