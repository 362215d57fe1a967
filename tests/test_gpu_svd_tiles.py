"""Truncated SVD at the edges of its kernels: bidiagonalisations of every number of rows per
block and beyond shared memory, spectra with multiplets, close pairs and zeros."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

import paper_2505_23429_gb300 as a2  # noqa: E402
from gpu_common import dev, host  # noqa: E402


def _check_svd(M, D):
    """Discarded weight, orthonormal P, and P S the projection of M on its range: singular
    values to 2^-40, vectors re-orthogonalised."""
    ctx = a2.Context(0)
    rows, cols = M.shape
    n = min(rows, cols)
    P = torch.zeros(rows * n, dtype=torch.float64, device="cuda")
    S = torch.zeros(n * cols, dtype=torch.float64, device="cuda")
    r, disc = a2.svd_split(ctx, dev(M.reshape(rows, 1, 1, cols)), D, 1e-12, P, S)
    Pm = host(P, ctx)[:rows * r].reshape(rows, r)
    Sm = host(S, ctx)[:r * cols].reshape(r, cols)
    s = np.linalg.svd(M, compute_uv=False)
    scale = np.linalg.norm(M)
    ref = np.linalg.norm(s[r:])
    assert r <= D
    assert abs(disc - ref) < 2e-12 * scale
    assert np.abs(Pm.T @ Pm - np.eye(r)).max() < 1e-12
    assert abs(np.linalg.norm(M - Pm @ Sm) - ref) < 2e-12 * scale
    ctx.close()


@pytest.mark.parametrize("rows,cols", [(1, 1), (2, 5), (33, 32), (144, 150), (145, 290), (310, 289),
                                       (20, 600), (600, 20), (433, 577), (9300, 6), (6, 9300)])
def test_svd_shapes(rows, cols):
    rng = np.random.default_rng(rows * 7 + cols)
    M = rng.standard_normal((rows, cols)) * 0.97 ** np.arange(cols)
    _check_svd(M, max(1, min(rows, cols) // 2))


# the values' interpolation needs them isolated: multiplets, pairs closer than the sample
# points, exact zeros and values far below the largest one take the other rounds
@pytest.mark.parametrize("kind", ["equal", "pairs", "close", "zeros", "graded"])
@pytest.mark.parametrize("n", [24, 150])
def test_svd_spectra(kind, n):
    rng = np.random.default_rng(n)
    s = 0.9 ** np.arange(n)
    if kind == "equal":
        s = np.ones(n)
    elif kind == "pairs":
        s = np.repeat(0.8 ** np.arange(n // 2), 2)
    elif kind == "close":
        s = np.sort(np.concatenate([s[::2], s[::2] * (1 + 1e-9)]))[::-1]
    elif kind == "zeros":
        s[n // 3:] = 0.0
    elif kind == "graded":
        s = np.logspace(0, -14, n)
    U, V = (np.linalg.qr(rng.standard_normal((n, n)))[0] for _ in range(2))
    _check_svd((U * s) @ V, n // 4)
