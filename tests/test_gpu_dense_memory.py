"""A dense expansion to the host gives its device memory back."""
import pytest

from paper_2403_01566_gb300 import inputs as I

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_2403_01566_gb300 import h2  # noqa: E402


def test_expansion_keeps_no_device_memory():
    w = I.grid_2d(64)
    A = h2.build(w.points, w.kernel_a, w.eta, w.leaf_size, w.order)
    A.matvec(w.points[:, 0].copy())  # (the cluster orders are on the device from here on)
    free = torch.cuda.mem_get_info()[0]
    A.to_dense()
    assert free - torch.cuda.mem_get_info()[0] < w.n * w.n * 8 // 4
