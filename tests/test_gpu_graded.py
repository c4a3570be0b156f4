"""Sliced tensor-core contractions of graded operands in the FP64 form: every
entry of a product within FP64's own bound, |y - A x| <= K 2^-53 |A| |x| for
sums of K terms, also where it is many orders below its row's and column's
largest entries.

One leaf of 64 points, so that y is one dense contraction of K = 64 (two chunks
of 32): a sliced chunk adds at most 2^-48.1 of its |A| |x| (see h2_gemm_tc.cu)
and two roundings, below 64 2^-53 = 2^-47.  The reference sums in extended
precision."""
import numpy as np
import pytest

from paper_2403_01566_gb300 import inputs as I

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_2403_01566_gb300 import h2  # noqa: E402

N = 64
POINTS = (np.arange(N) / N).reshape(N, 1)


def _gauss(width):
    """exp(-r^2 / width): down to 1e-16 of the diagonal 15 points away, and no
    subnormal entries (whose rows take the plain FP64 sum) 63 points away."""
    A = h2.build(POINTS, I.KernelSpec(I.KERNEL_GAUSS, 1.0, 1.0, width), 2.0, N, 4)
    return A, A.to_dense()


def _worst(y, A, x):
    """Largest error of an entry of A x, in units of 2^-53 (|A| |x|)."""
    Al, xl = A.astype(np.longdouble), x.astype(np.longdouble)
    err, ref = np.abs(y.astype(np.longdouble) - Al @ xl), np.abs(Al) @ np.abs(xl)
    assert np.array_equal(y[ref == 0], np.zeros(int((ref == 0).sum())))
    return float((err[ref > 0] / ref[ref > 0]).max() * 2.0 ** 53)


@pytest.mark.parametrize("nrhs", [1, 8, 64, 65])
@pytest.mark.parametrize("peak", [1e6, 1e12, 1e16])
def test_vectors_with_one_large_entry(nrhs, peak):
    A, Ad = _gauss(0.00145)
    x = np.random.default_rng(3).standard_normal((N, nrhs))
    x[np.arange(nrhs) % N, np.arange(nrhs)] *= peak
    x[5] *= peak
    assert _worst(A.matvec_batch(x), Ad, x) <= N


@pytest.mark.parametrize("precision", [0, 2])
def test_product_of_narrow_gaussians(precision):
    (A, Ad), (B, Bd) = _gauss(0.00145), _gauss(0.002)
    assert _worst(h2.mul(A, B, 1e-6, precision=precision).to_dense(), Ad, Bd) <= N
