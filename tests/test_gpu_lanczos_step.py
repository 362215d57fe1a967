"""The fused Lanczos step over vector lengths, Krylov sizes and spectra: two-site chains
H = A (x) 1 + 1 (x) B, whose one local problem is the whole chain and whose lowest
eigenvalue is the sum of those of A and B."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

import paper_2505_23429_gb300 as a2  # noqa: E402

EIG_TOL = 1e-10


def _site(n, shift, close, rng):
    """Tridiagonal symmetric, lowest levels well separated, or two of them `close` apart."""
    d = shift + np.linspace(0.0, 3.0, n) + (np.arange(n) > 0) * 1.0
    if close and n > 2:
        d[1] = d[0] + close
    off = 0.1 * rng.uniform(0.5, 1.0, max(n - 1, 0))
    if close and n > 2:
        off[:2] = 0.0
    return np.diag(d) + np.diag(off, 1) + np.diag(off, -1)


def _lowest(n, max_krylov, shift=0.0, close=0.0, scale=1.0):
    rng = np.random.default_rng(n)
    A, B = (scale * _site(n, s, close, rng) for s in (shift, -0.3))
    W0 = np.zeros((1, n, n, 2))
    W1 = np.zeros((2, n, n, 1))
    W0[0, :, :, 0], W0[0, :, :, 1] = A, np.eye(n)
    W1[0, :, :, 0], W1[1, :, :, 0] = np.eye(n), B
    ctx = a2.Context(0)
    mpo = a2.MPO(ctx, [W0, W1])
    r0 = min(n, 3)
    t = a2.TT.from_cores(ctx, [rng.standard_normal((1, n, r0)), rng.standard_normal((r0, n, 1))])
    t.left_orthogonalize()
    r = a2.additive_sweep(ctx, t, mpo, 1, D_max=4, eig_tol=EIG_TOL, svd_tol=1e-12,
                          max_krylov=max_krylov, max_restarts=2000, prec="fp64")
    ref = np.linalg.eigvalsh(A)[0] + np.linalg.eigvalsh(B)[0]
    assert r["unconverged"] == 0
    ctx.close()
    return r["energy_local"][0], ref


# a Ritz value is within the residual EIG_TOL * max(1, |theta|) of an eigenvalue; the start
# vector has weight on the lowest one
@pytest.mark.parametrize("max_krylov", [2, 3, 20, 63])
@pytest.mark.parametrize("n", [1, 2, 5, 11, 12, 36, 70])
def test_sizes_and_krylov_dims(n, max_krylov):
    th, ref = _lowest(n, max_krylov)
    assert abs(th - ref) <= 2 * EIG_TOL * max(1.0, abs(ref))


# slices beyond one entry per thread; beyond shared memory (kept in device memory)
@pytest.mark.parametrize("n", [400, 1800])
def test_long_vectors(n):
    th, ref = _lowest(n, 40)
    assert abs(th - ref) <= 2 * EIG_TOL * max(1.0, abs(ref))


# two lowest levels closer than the sample points of the fast tridiagonal solver; large
# shifts; scales outside the FP32 range of its first phase
@pytest.mark.parametrize("kw", [dict(close=1e-9), dict(close=1e-7), dict(shift=1e4),
                                dict(shift=-1e4), dict(scale=1e18), dict(scale=1e-3)])
def test_spectra(kw):
    th, ref = _lowest(24, 30, **kw)
    assert abs(th - ref) <= 2 * EIG_TOL * max(1.0, abs(ref)) + 2e-9 * (kw.get("close", 0) > 0)
