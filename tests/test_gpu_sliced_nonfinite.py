"""Operands that the BF16 slices cannot hold (NaN, infinities, entries beyond the FP32 range)
reach every output that depends on them, and no other, beyond the first 256-entry chunk of
the reduction and through both slicing kernels."""
import numpy as np
import pytest

from oracle.env import env_left_update as oracle_left
from oracle.env import heff_apply as oracle_heff
from synthetic import heisenberg_mpo

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

import paper_2505_23429_gb300 as a2  # noqa: E402
from gpu_common import dev, host  # noqa: E402

J = 5


def _check(got, oracle, arrays, name, at):
    """arrays: operands by name; the outputs that depend on element `at` of `name` (with the
    cores' zeros; at most with dense cores, as NaN times zero is NaN)."""
    hit = {k: np.abs(v) for k, v in arrays.items()}
    hit[name] = np.zeros_like(hit[name])
    hit[name][at] = 1.0
    must = oracle(**hit) > 0.0
    may = oracle(**{k: np.ones_like(v) if k[0] == "W" else v for k, v in hit.items()}) > 0.0
    bad = ~np.isfinite(got)
    assert must.any() and bad[must].all()
    assert not bad[~may].any()


@pytest.mark.parametrize("value", [np.nan, np.inf, -1e200, 1e39])
@pytest.mark.parametrize("name,at", [("H", (7, 1, 300)), ("bra", (290, 1, 9)),
                                     ("ket", (300, 0, 9))])
def test_env_update(name, at, value):
    m = heisenberg_mpo(12)
    rng = np.random.default_rng(1)
    Dl, Dr = 520, 64
    ops = dict(H=rng.standard_normal((Dl, 5, Dl)), bra=rng.standard_normal((Dl, 2, Dr)), W=m[J],
               ket=rng.standard_normal((Dl, 2, Dr)))
    dirty = {k: v.copy() for k, v in ops.items()}
    dirty[name][at] = value
    ctx = a2.Context(0)
    out = torch.zeros((Dr, 5, Dr), dtype=torch.float64, device="cuda")
    a2.env_update(ctx, a2.MPO(ctx, m), J, 0, dev(dirty["H"]), dev(dirty["bra"]), dev(dirty["ket"]),
                  out, prec="f64emu")
    _check(host(out, ctx), lambda H, bra, W, ket: oracle_left(H, bra, W, ket), ops, name, at)
    ctx.close()


@pytest.mark.parametrize("value", [np.nan, -np.inf, 1e200, 1e39])
@pytest.mark.parametrize("name,at", [("L", (3, 2, 280)), ("R", (5, 4, 70)), ("x", (299, 1, 0, 7))])
def test_heff(name, at, value):
    m = heisenberg_mpo(12)
    rng = np.random.default_rng(2)
    Dl, Dr = 300, 72
    ops = dict(L=rng.standard_normal((Dl, 5, Dl)), W1=m[J], W2=m[J + 1],
               R=rng.standard_normal((Dr, 5, Dr)), x=rng.standard_normal((Dl, 2, 2, Dr)))
    dirty = {k: v.copy() for k, v in ops.items()}
    dirty[name][at] = value
    ctx = a2.Context(0)
    y = torch.zeros(ops["x"].shape, dtype=torch.float64, device="cuda")
    a2.heff_apply(ctx, a2.MPO(ctx, m), J, dev(dirty["L"]), dev(dirty["R"]), dev(dirty["x"]), y,
                  prec="f64emu")
    _check(host(y, ctx), lambda L, W1, W2, R, x: oracle_heff(L, W1, W2, R, x), ops, name, at)
    ctx.close()
