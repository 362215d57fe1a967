"""LQ at the edges of its kernels: rows around the 32-row panels, widths around the cluster
sizes and beyond the shared-memory path."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

import paper_2505_23429_gb300 as a2  # noqa: E402
from gpu_common import dev, host  # noqa: E402

EPS = 2.0 ** -53


# Householder LQ: ||A - L Q||_F and the entries of Q Q^T - 1 stay below c k eps (Higham,
# Accuracy and Stability of Numerical Algorithms, Th. 19.4), c = 8
@pytest.mark.parametrize("rows,cols", [(31, 40), (32, 33), (33, 300), (65, 64), (96, 97), (160, 31),
                                       (130, 1030), (300, 700), (40, 5000), (35, 9150),
                                       (34, 9300)])
def test_lq(rows, cols):
    ctx = a2.Context(0)
    M = np.random.default_rng(rows + cols).standard_normal((rows, cols))
    k = min(rows, cols)
    L = torch.zeros((rows, k), dtype=torch.float64, device="cuda")
    Q = torch.zeros((k, cols), dtype=torch.float64, device="cuda")
    a2.lq(ctx, dev(M), L, Q)
    L, Q = host(L, ctx), host(Q, ctx)
    tol = 8 * max(k, 4) * 2 * EPS
    assert np.linalg.norm(L @ Q - M) < tol * np.linalg.norm(M)
    assert np.abs(Q @ Q.T - np.eye(k)).max() < tol
    assert np.all(np.diag(L) >= 0.0) and np.abs(np.triu(L, 1)).max() == 0.0
    ctx.close()


# a NaN in a row reaches that row of Q, in the first panel and in a later one
@pytest.mark.parametrize("cols", [64, 9300])
@pytest.mark.parametrize("row", [5, 37])
def test_lq_nan_is_visible(row, cols):
    ctx = a2.Context(0)
    M = np.random.default_rng(1).standard_normal((40, cols))
    M[row, 50] = np.nan
    L = torch.zeros((40, 40), dtype=torch.float64, device="cuda")
    Q = torch.zeros((40, cols), dtype=torch.float64, device="cuda")
    a2.lq(ctx, dev(M), L, Q)
    assert np.isnan(host(Q, ctx)[row]).any()
    ctx.close()
