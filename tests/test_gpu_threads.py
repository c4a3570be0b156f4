"""One handle used by several host threads at once (ctypes calls release the
interpreter lock): every thread gets what a single one gets."""
import threading

import numpy as np
import pytest

from paper_2403_01566_gb300 import inputs as I

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_2403_01566_gb300 import h2  # noqa: E402

THREADS = 4


def _at_once(f):
    """f(i) on THREADS threads that start together; their results."""
    out, gate = [None] * THREADS, threading.Barrier(THREADS)

    def work(i):
        gate.wait()
        out[i] = f(i)

    ts = [threading.Thread(target=work, args=(i,)) for i in range(THREADS)]
    for t in ts:
        t.start()
    for t in ts:
        t.join()
    return out


@pytest.mark.parametrize("mul", [h2.mul, h2.mul_h], ids=["mul", "mul_h"])
def test_dense_expansion_of_a_fresh_product(mul):
    """The first expansions of a product, by all threads at once."""
    w = I.square_2d(700, seed=3)
    A = h2.build(w.points, w.kernel_a, w.eta, w.leaf_size, w.order)
    B = h2.build(w.points, w.kernel_b, w.eta, w.leaf_size, w.order)
    for _ in range(3):
        C = mul(A, B, 1e-6)
        got = _at_once(lambda i: C.to_dense())
        want = C.to_dense()
        for g in got:
            assert g is not None and np.array_equal(g, want)


@pytest.mark.parametrize("nrhs", [1, 8])
def test_matrix_vector_products_at_once(nrhs):
    """Threads multiply two products of one structure, which share a plan, its
    workspace and its rank slots."""
    w = I.square_2d(700, seed=3)
    A = h2.build(w.points, w.kernel_a, w.eta, w.leaf_size, w.order)
    B = h2.build(w.points, w.kernel_b, w.eta, w.leaf_size, w.order)
    Cs = [h2.mul(A, B, 1e-6), h2.mul(B, A, 1e-2)]
    X = np.random.default_rng(1).standard_normal((THREADS, w.n, nrhs))
    want = [Cs[i % 2].matvec_batch(X[i]) for i in range(THREADS)]
    res = _at_once(lambda i: [Cs[i % 2].matvec_batch(X[i]) for _ in range(50)])
    for i in range(THREADS):
        assert all(np.array_equal(y, want[i]) for y in res[i])


def test_products_at_once():
    """Threads run products of one structure and other operands: one plan
    instance, its header and its workspace."""
    w = I.square_2d(700, seed=3)
    A = h2.build(w.points, w.kernel_a, w.eta, w.leaf_size, w.order)
    B = h2.build(w.points, w.kernel_b, w.eta, w.leaf_size, w.order)
    pairs = [(A, B), (B, A), (A, A), (B, B)]
    want = [h2.mul(x, y, 1e-6).to_dense() for x, y in pairs]
    res = _at_once(lambda i: [h2.mul(*pairs[i], 1e-6).to_dense() for _ in range(3)])
    for i in range(THREADS):
        assert all(np.array_equal(c, want[i]) for c in res[i])
