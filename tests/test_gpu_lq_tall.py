"""LQ on both sides of the lines between panels and the cooperative kernel: many more rows than
columns, around 48, 96, 200, 320 and 480 columns."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

import paper_2505_23429_gb300 as a2  # noqa: E402
from gpu_common import dev, host  # noqa: E402

EPS = 2.0 ** -53


def _lq(M):
    ctx = a2.Context(0)
    rows, cols = M.shape
    k = min(rows, cols)
    L = torch.zeros((rows, k), dtype=torch.float64, device="cuda")
    Q = torch.zeros((k, cols), dtype=torch.float64, device="cuda")
    a2.lq(ctx, dev(M), L, Q)
    L, Q = host(L, ctx), host(Q, ctx)
    assert a2.device_error(ctx) == 0
    ctx.close()
    return L, Q


# Householder LQ: ||A - L Q||_F and the entries of Q Q^T - 1 stay below c k eps (Higham,
# Accuracy and Stability of Numerical Algorithms, Th. 19.4), c = 8
@pytest.mark.parametrize("rows,cols", [(752, 47), (768, 48), (1519, 95), (1520, 95), (383, 96),
                                       (384, 96), (796, 199), (599, 200), (600, 200),
                                       (959, 320), (960, 320), (1925, 321), (1926, 321),
                                       (2874, 479), (1920, 480), (5000, 100)])
def test_lq(rows, cols):
    M = np.random.default_rng(rows + cols).standard_normal((rows, cols))
    M *= 10.0 ** -np.linspace(0.0, 3.0, rows)[:, None]
    L, Q = _lq(M)
    tol = 8 * cols * 2 * EPS
    assert np.linalg.norm(L @ Q - M) < tol * np.linalg.norm(M)
    assert np.abs(Q @ Q.T - np.eye(cols)).max() < tol
    assert np.all(np.diag(L) >= 0.0) and np.abs(np.triu(L, 1)).max() == 0.0


def test_nan_and_zero_rows():
    M = np.random.default_rng(3).standard_normal((700, 128))
    M[20] = 0.0                                  # no reflection: its row of Q is a unit vector
    L, Q = _lq(M)
    assert np.linalg.norm(L @ Q - M) < 8 * 128 * 2 * EPS * np.linalg.norm(M)
    assert L[20, 20] == 0.0
    M[37, 50] = np.nan
    assert np.isnan(_lq(M)[1][37]).any()
