"""Outputs of split trees: even and odd nodes per leaf, aligned and odd output addresses and page-locked host memory all
receive the same bits."""
import numpy as np
import pytest

import paper_1908_07392_gb300 as V
from paper_1908_07392_gb300 import inputs as I

pytestmark = pytest.mark.gpu


# p = 2 .. 16: 12 to 768 rows a destination (one field's end inside a warp's rows, and at their edge); 1 leaf and many
@pytest.mark.parametrize("depth,p", [(0, 2), (0, 3), (2, 2), (3, 3), (2, 5), (2, 7), (3, 8), (2, 11), (2, 13), (2, 15), (2, 16)])
def test_outputs_at_any_address(depth, p):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    vp = V.VolumePotential(1, 12.0, p, I.uniform_tree(depth, side=2.0), precision=V.VP_PREC_SPLIT)
    try:
        n = vp.N
        f = torch.from_numpy(np.random.default_rng(p).standard_normal(n))
        fd = f.cuda()
        u, g = (t.cpu() for t in vp(fd))
        assert torch.isfinite(u).all() and torch.isfinite(g).all() and (u != 0).any()
        for off in (1, 2, 3):
            bu = torch.full((n + 4,), 7.0, dtype=torch.float64, device="cuda")
            bg = torch.full((2 * n + 4,), 7.0, dtype=torch.float64, device="cuda")
            V.vp_eval(vp.tree, fd, bu[off:off + n], bg[off:off + 2 * n])
            assert torch.equal(bu[off:off + n].cpu(), u) and torch.equal(bg[off:off + 2 * n].view(2, n).cpu(), g)
            for b, m in ((bu, n), (bg, 2 * n)):   # nothing beside the outputs is written
                assert (b[:off] == 7.0).all() and (b[off + m:] == 7.0).all()
        hu, hg = torch.empty(n, dtype=torch.float64).pin_memory(), torch.empty(2, n, dtype=torch.float64).pin_memory()
        V.vp_eval_host(vp.tree, f.pin_memory(), hu, hg)
        assert torch.equal(hu, u) and torch.equal(hg, g)
    finally:
        vp.close()
