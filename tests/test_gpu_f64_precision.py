"""FP64 contraction tiles to FP64's own error: against the CPU oracle at 1e-10 where the expansion order resolves it, and,
for the low orders, linearity, which an intermediate rounded below FP64 would break."""
import numpy as np
import pytest

import paper_1908_07392_gb300 as V
from paper_1908_07392_gb300 import inputs as I
from gpu_util import TOL_FP64, gpu_eval, oracle_eval, rel_err, sample_nodes

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    V.load_library()


def tree_of(kind, seed):
    if kind.startswith("uniform"):
        return I.uniform_tree(int(kind[7:]), side=2.0)
    return I.random_balanced_tree(np.random.default_rng(seed), 25, 6)


def field(tree, p, a=-4.0, b=5.0):
    X, Y = I.node_coords(tree, p)
    return np.exp(a * ((X - 0.1) ** 2 + (Y + 0.2) ** 2)) * (1 + 0.3 * np.sin(b * X))


@pytest.mark.parametrize("kernel,p,order,kind", [(0, 13, 40, "random"), (1, 16, 40, "uniform3"), (0, 16, 60, "random"),
                                                 (0, 6, 40, "uniform5"), (0, 4, 40, "uniform0"), (1, 9, 40, "uniform4")])
def test_against_the_oracle(kernel, p, order, kind):
    tree = tree_of(kind, p)
    w = I.Workload("tiles", kernel, 15.0, p, tree, field(tree, p))
    idx = sample_nodes(w, 60, p)
    for got, ref in zip(gpu_eval(w, order=order), oracle_eval(w, idx)):
        assert rel_err(got[idx], ref) <= TOL_FP64


# sums of a few thousand terms, each rounded to 2^-53, that cancel to a hundredth of their magnitudes at worst
@pytest.mark.parametrize("kernel,p,order,kind", [(0, 2, 4, "uniform2"), (0, 3, 7, "random"), (1, 5, 11, "uniform3"),
                                                 (1, 7, 23, "random"), (0, 9, 33, "uniform5")])
def test_linearity(kernel, p, order, kind):
    tree = tree_of(kind, p)
    f, g = field(tree, p), field(tree, p, -1.0, 3.0)
    one, two, both = (gpu_eval(I.Workload("tiles", kernel, 15.0, p, tree, s), order=order) for s in (f, g, f + g))
    for a, b, c in zip(one, two, both):
        assert np.abs(a + b - c).max() <= 1e-12 * np.abs(c).max()
