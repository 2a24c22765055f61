"""The FP64 contraction's tiles at their edges (rows and columns that are no multiple of 8 and 4, K that is no
multiple of 16 or 4, the panel kernel up to its largest K, launches on both sides of the line between the two
kernels): FP64 evaluations against split-precision ones of the same tables, which share none of that code, to
the split form's stated error."""
import numpy as np
import pytest

import paper_1908_07392_gb300 as V
from paper_1908_07392_gb300 import inputs as I

pytestmark = pytest.mark.gpu

TOL_SPLIT = 1e-9


def tree_of(kind, seed):
    if kind.startswith("uniform"):
        return I.uniform_tree(int(kind[7:]), side=2.0)
    return I.random_balanced_tree(np.random.default_rng(seed), 25, 6)


@pytest.mark.parametrize("kernel,p,order,kind", [(0, 2, 4, "uniform2"), (0, 3, 7, "random"), (1, 5, 11, "uniform3"),
                                                 (1, 7, 23, "random"), (0, 13, 40, "random"), (1, 16, 40, "uniform3"),
                                                 (0, 16, 60, "random"), (0, 6, 40, "uniform5"), (0, 9, 33, "uniform5"),
                                                 (0, 4, 20, "uniform0")])
def test_fp64_against_split(kernel, p, order, kind):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    tree = tree_of(kind, p)
    X, Y = I.node_coords(tree, p)
    f = torch.from_numpy(np.exp(-4 * ((X - 0.1) ** 2 + (Y + 0.2) ** 2)) * (1 + 0.3 * np.sin(5 * X))).cuda()
    res = []
    for precision in (V.VP_PREC_FP64, V.VP_PREC_SPLIT):
        vp = V.VolumePotential(kernel, 15.0, p, tree, order=order, precision=precision)
        try:
            u, g = vp(f)
            torch.cuda.synchronize()
            res.append([u.cpu().numpy(), g[0].cpu().numpy(), g[1].cpu().numpy()])
        finally:
            vp.close()
    for a, b in zip(*res):
        assert np.abs(a - b).max() <= TOL_SPLIT * np.abs(b).max()
