"""Boundary evaluation with one and with two targets per block (chosen by the number of targets): both sides of the
line, odd numbers, Bessel and algebraic pairs. A target's sum does not depend on the others beyond its rounding."""
import numpy as np
import pytest

import paper_1908_07392_gb300 as V

pytestmark = pytest.mark.gpu


# each target alone takes the one-target form; the terms are the same in both forms, at most 16 of them meet in a thread,
# then 5 + 8 partial sums: 2 (16 + 13) 2^-53 of the sum of their magnitudes, each below |m| w / r with r >= 0.2 here
@pytest.mark.parametrize("alpha", [8.0, 100.0, 400.0])
def test_targets_together_and_alone(alpha):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    b = V.BIE(alpha, phase=0.1, n_panels=64, max_krylov=1)
    try:
        sms = torch.cuda.get_device_properties(0).multi_processor_count
        rng = np.random.default_rng(3)
        M = 4 * sms + 1
        r, th = 0.5 * np.sqrt(rng.uniform(0, 1, M)), rng.uniform(0, 2 * np.pi, M)
        xy = torch.from_numpy(np.stack([r * np.cos(th), r * np.sin(th)])).cuda()
        mu = torch.from_numpy(rng.standard_normal(2 * b.N)).cuda()
        alone = torch.cat([b.eval(mu, xy[:, k:k + 1].contiguous()) for k in range(M)], dim=1)
        mag = (mu.view(-1, 2).abs().sum(1) * b.nodes[4]).sum() / 0.2
        for m in (1, 2, sms, 2 * sms - 1, 2 * sms, 2 * sms + 1, 3 * sms, 3 * sms + 1, 4 * sms - 1, 4 * sms, M):
            u = b.eval(mu, xy[:, :m].contiguous())
            assert float((u - alone[:, :m]).abs().max()) <= 58 * 2.0 ** -53 * float(mag)
    finally:
        b.close()
