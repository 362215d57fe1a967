"""The Lanczos step's parts by themselves: its grid barrier that runs out (without a GPU fault:
one arrival too many is expected, with a short limit), and its tridiagonal solver on both of its
paths against LAPACK."""
import numpy as np
import pytest

from synthetic import heisenberg_mpo, random_tt_cores

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

import paper_2505_23429_gb300 as a2  # noqa: E402

A2_ETIMEOUT = -6
EPS = 2.0 ** -52


@pytest.fixture(scope="module")
def ctx():
    c = a2.Context(0)
    yield c
    c.close()


def test_barrier_gives_up_and_the_next_solve_works(ctx):
    mpo = a2.MPO(ctx, heisenberg_mpo(6))

    def solve():
        t = a2.TT.from_cores(ctx, random_tt_cores([2] * 6, 4, 3))
        t.left_orthogonalize()
        r = a2.additive_sweep(ctx, t, mpo, 1, D_max=8, eig_tol=1e-10, svd_tol=1e-12, prec="fp64")
        assert r["unconverged"] == 0
        return np.array(r["energy_local"])

    before = solve()
    for _ in range(2):
        assert a2.selftest_lanczos_timeout(ctx) == A2_ETIMEOUT
        assert "gave up" in a2.last_error(ctx)
        assert a2.device_error(ctx) == 0                   # not an error word of the GEMMs
    assert np.abs(solve() - before).max() < 1e-9 * np.abs(before).max()


def _tri(kind, k, rng):
    a, b = rng.standard_normal(k), rng.uniform(0.2, 1.0, k - 1)
    if kind == "lanczos":              # a Krylov matrix: the lowest value is isolated
        q, _ = np.linalg.qr(rng.standard_normal((2 * k + 8, k)))
        lam = np.concatenate([[-3.0], np.linspace(0.0, 5.0, 2 * k + 7)])
        a, b, v, w = [], [], np.full(2 * k + 8, (2 * k + 8) ** -0.5), None
        basis = [v]
        for _ in range(k):
            w = lam * basis[-1]
            a.append(basis[-1] @ w)
            for _ in range(2):
                for u in basis:
                    w = w - (u @ w) * u
            b.append(np.linalg.norm(w))
            basis.append(w / b[-1])
        a, b = np.array(a), np.array(b[:-1])
    elif kind == "shifted":            # the levels in the last 2^-20 of the scale
        a = a + 1e6
    elif kind == "tiny":
        a, b = 1e-100 * a, 1e-100 * b
    elif kind == "huge":
        a, b = 1e100 * a, 1e100 * b
    elif kind == "graded":
        a, b = a * 10.0 ** -np.linspace(0, 12, k), b * 10.0 ** -np.linspace(0, 12, k)[1:]
    elif kind == "zeros":
        b = b * (rng.random(k - 1) < 0.7)
    return a, b


def _scale(a, b):
    r = np.abs(a).copy()
    r[:-1] += np.abs(b)
    r[1:] += np.abs(b)
    return r.max()


# eigenvalue: k roundings of the scale; residual: what the fast method accepts
def _check(ctx, a, b, tol=None):
    th, z, general = a2.tridiag_lowest(ctx, a, b)
    T = np.diag(a) + np.diag(b, 1) + np.diag(b, -1)
    sc, k = _scale(a, b), len(a)
    ref = np.linalg.eigvalsh(T / sc)[0] * sc
    assert abs(th - ref) <= (tol or 4 * max(k, 4) * EPS * sc)
    assert abs(np.linalg.norm(z) - 1.0) <= 4 * max(k, 4) * EPS
    assert np.linalg.norm((T / sc) @ z - (th / sc) * z) <= 2e-12
    return general


@pytest.mark.parametrize("kind", ["random", "lanczos", "shifted", "tiny", "huge", "graded", "zeros"])
def test_tridiagonal(ctx, kind):
    rng = np.random.default_rng(5)
    ran = [_check(ctx, *_tri(kind, k, rng)) for k in range(1, 64)]
    if kind == "lanczos":
        assert not any(ran)                                # the fast path is the one that runs
    if kind in ("tiny", "huge"):
        assert all(ran[1:])


@pytest.mark.parametrize("gap", [1e-7, 1e-9, 1e-11])
@pytest.mark.parametrize("k", [3, 24, 63])
def test_close_levels(ctx, k, gap):
    """Two lowest levels `gap` apart: the returned one is the lower, to a hundredth of it."""
    a = 1.0 + np.linspace(0.0, 1.0, k)
    b = 0.05 * np.ones(k - 1)
    a[0], a[1], b[:2] = 0.0, gap, 0.0
    for a[0], a[1] in ((0.0, gap), (gap, 0.0)):
        general = _check(ctx, a, b, 0.01 * gap)
        assert general or gap > 1e-8                       # closer than 1e-8 of the scale
