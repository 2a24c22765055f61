"""The far-field chain of split trees beside the near field, its launches overlapping or not (chosen by the number of
nodes), against the same evaluation launch by launch on one stream: the same bits, repeatedly."""
import numpy as np
import pytest

import paper_1908_07392_gb300 as V
from paper_1908_07392_gb300 import inputs as I

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("kernel,p,depth", [(1, 4, 2), (0, 8, 4), (1, 12, 6), (0, 16, 6), (1, 11, 7)])  # 256 .. 1.98M nodes
def test_overlapped_against_in_order(kernel, p, depth):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    vp = V.VolumePotential(kernel, 25.0, p, I.uniform_tree(depth, side=2.0), precision=V.VP_PREC_SPLIT)
    try:
        for seed in range(3):
            f = torch.from_numpy(np.random.default_rng(seed).standard_normal(vp.N)).cuda()
            u, g = torch.empty_like(f), torch.empty(2, vp.N, dtype=torch.float64, device="cuda")
            V.vp_eval_timed(vp.tree, f, u, g)
            for _ in range(4):
                u2, g2 = vp(f)
                assert torch.equal(u, u2) and torch.equal(g, g2)
    finally:
        vp.close()
