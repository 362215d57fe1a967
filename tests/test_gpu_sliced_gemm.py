"""Tensor-core products of split operands: reductions around the 32-element blocks and the
256-element chunks with their own exponents, rows and columns around the 128-row and
256-column tiles, operands of very uneven scales, against the oracle."""
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
from gpu_common import dev, host, rel  # noqa: E402

# unit roundoff times the square root of at most 5 * 520 products, a few stages
TOL = {"f32emu": 1e-5, "f64emu": 1e-13}


@pytest.mark.parametrize("prec", ["f32emu", "f64emu"])
@pytest.mark.parametrize("Dl,Dr", [(31, 33), (32, 255), (257, 8), (63, 513), (300, 52), (512, 64)])
def test_heff_around_blocks(prec, Dl, Dr):
    ctx = a2.Context(0)
    m = heisenberg_mpo(12)
    mpo = a2.MPO(ctx, m)
    rng = np.random.default_rng(Dl * 1000 + Dr)
    Lh = rng.standard_normal((Dl, 5, Dl))
    Rh = rng.standard_normal((Dr, 5, Dr))
    x = rng.standard_normal((Dl, 2, 2, Dr))
    y = torch.zeros(x.shape, dtype=torch.float64, device="cuda")
    a2.heff_apply(ctx, mpo, 5, dev(Lh), dev(Rh), dev(x), y, prec=prec)
    assert rel(host(y, ctx), oracle_heff(Lh, m[5], m[6], Rh, x)) < TOL[prec]
    assert a2.device_error(ctx) == 0
    ctx.close()


# entries spread over 2^+-40 along the reduction index: the slices of one chunk end 2^-55
# below its largest entry, so the error stays at rounding of the largest terms of the sum
@pytest.mark.parametrize("Dl,Dr", [(250, 31), (260, 64), (520, 24)])
def test_env_update_uneven_scales(Dl, Dr):
    ctx = a2.Context(0)
    m, j = heisenberg_mpo(12), 5
    mpo = a2.MPO(ctx, m)
    rng = np.random.default_rng(Dl)
    Hin = rng.standard_normal((Dl, 5, Dl))
    bra = rng.standard_normal((Dl, 2, Dr))
    ket = rng.standard_normal((Dl, 2, Dr)) * 2.0 ** rng.integers(-40, 40, Dl)[:, None, None]
    out = torch.zeros((Dr, 5, Dr), dtype=torch.float64, device="cuda")
    a2.env_update(ctx, mpo, j, 0, dev(Hin), dev(bra), dev(ket), out, prec="f64emu")
    ref = oracle_left(Hin, bra, m[j], ket)
    mag = oracle_left(abs(Hin), abs(bra), abs(m[j]), abs(ket))
    assert np.max(np.abs(host(out, ctx) - ref) / mag.max()) < TOL["f64emu"]
    ctx.close()
