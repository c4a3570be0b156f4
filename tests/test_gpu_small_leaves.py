"""Leaves of two points with k = 64: the tensor-core form's smallest tiles (2
rows by 64 columns), whose slices fill most of a launch's shared memory.
Every admissible block of the product has to be within eps of the exact one."""
import numpy as np
import pytest

from oracle import h2oracle as O
from paper_2403_01566_gb300 import inputs as I
from tests.oracle_cases import build_pair

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_2403_01566_gb300 import h2  # noqa: E402


@pytest.mark.parametrize("precision", [0, 3, 4])
@pytest.mark.parametrize("w", [I.square_2d(64, seed=7, leaf=2, order=8), I.cube_3d(64, seed=7, leaf=2, order=4)],
                         ids=lambda w: w.name)
def test_leaves_of_two_points(w, precision):
    eps = 1e-4
    A = h2.build(w.points, w.kernel_a, w.eta, w.leaf_size, w.order)
    B = h2.build(w.points, w.kernel_b, w.eta, w.leaf_size, w.order)
    C = h2.mul(A, B, eps, precision=precision, max_rank=64).to_dense()
    X, Y = build_pair(w)
    Z = X.dense() @ Y.dense()
    for b in O.block_leaves(X.blocks):
        ix = np.ix_(b.t.idx, b.s.idx)
        assert np.linalg.norm(C[ix] - Z[ix], 2) <= eps * np.linalg.norm(Z[ix], 2)
