"""Sparse MPO rows staged in shared memory: the operator at vector lengths below, at and
around the slice widths (2 to 64 elements a lane group), aligned and odd, in the three
tensor-core precisions, against the oracle."""
import numpy as np
import pytest

from oracle.env import env_left_update as oracle_left
from oracle.env import heff_apply as oracle_heff
from synthetic import chemistry_integrals, chemistry_mpo

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

import paper_2505_23429_gb300 as a2  # noqa: E402
from gpu_common import dev, host, rel  # noqa: E402

# unit roundoffs 2^-9 (BF16 intermediates, four stages), 2^-24 and 2^-53 times the square
# root of the few thousand products of an element
TOL = {"bf16": 2e-2, "f32emu": 5e-6, "f64emu": 1e-13}


@pytest.fixture(scope="module")
def chem10():
    return chemistry_mpo(*chemistry_integrals(10, 2505))


@pytest.mark.parametrize("prec", ["bf16", "f32emu", "f64emu"])
@pytest.mark.parametrize("k,Dl,Dr", [(3, 1, 1), (3, 3, 7), (4, 8, 4), (4, 16, 33), (5, 5, 64),
                                     (2, 40, 72), (6, 17, 130)])
def test_heff(chem10, prec, k, Dl, Dr):
    ctx = a2.Context(0)
    m = chem10
    mpo = a2.MPO(ctx, m)
    rng = np.random.default_rng(100 * Dl + Dr)
    Lh = rng.standard_normal((Dl, m[k].shape[0], Dl))
    Rh = rng.standard_normal((Dr, m[k + 1].shape[3], Dr))
    x = rng.standard_normal((Dl, m[k].shape[1], m[k + 1].shape[1], Dr))
    y = torch.zeros(x.shape, dtype=torch.float64, device="cuda")
    a2.heff_apply(ctx, mpo, k, dev(Lh), dev(Rh), dev(x), y, prec=prec)
    got = host(y, ctx)
    assert a2.device_error(ctx) == 0
    assert rel(got, oracle_heff(Lh, m[k], m[k + 1], Rh, x)) < TOL[prec]
    ctx.close()


@pytest.mark.parametrize("Dl,Dr", [(6, 9), (24, 31), (32, 64)])
def test_env_update(chem10, Dl, Dr):
    ctx = a2.Context(0)
    m, j = chem10, 4
    mpo = a2.MPO(ctx, m)
    rng = np.random.default_rng(Dl)
    Hin = rng.standard_normal((Dl, m[j].shape[0], Dl))
    bra = rng.standard_normal((Dl, m[j].shape[1], Dr))
    ket = rng.standard_normal((Dl, m[j].shape[2], Dr))
    out = torch.zeros((Dr, m[j].shape[3], Dr), dtype=torch.float64, device="cuda")
    a2.env_update(ctx, mpo, j, 0, dev(Hin), dev(bra), dev(ket), out, prec="f64emu")
    got = host(out, ctx)
    assert rel(got, oracle_left(Hin, bra, m[j], ket)) < TOL["f64emu"]
    ctx.close()
