"""Truncated SVD on both sides of the line between the bidiagonalisation's single blocks and its
clusters: around 128 columns, and where fewer blocks would cost the warps another round."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

from test_gpu_svd_tiles import _check_svd  # noqa: E402


@pytest.mark.parametrize("rows,cols", [(128, 128), (129, 129), (128, 1220), (129, 1220),
                                       (1150, 130), (1160, 130), (4000, 129), (130, 9300),
                                       (7, 8), (8, 8), (140, 129)])
def test_svd_shapes(rows, cols):
    rng = np.random.default_rng(rows * 11 + cols)
    n = min(rows, cols)
    M = rng.standard_normal((rows, n)) * 0.97 ** np.arange(n) @ rng.standard_normal((n, cols))
    _check_svd(M, max(1, n // 2))
