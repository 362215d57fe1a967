"""SIMT GEMM tiles: the operator at sizes around every tile edge (8, 16, 32, 64; 128 in
FP32) and around the lines where the choice changes, against the oracle."""
import numpy as np
import pytest

from oracle.env import heff_apply as oracle_heff
from synthetic import heisenberg_mpo

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

import paper_2505_23429_gb300 as a2  # noqa: E402
from gpu_common import dev, host, rel  # noqa: E402

# sums of at most 5 * 400 products: eps * sqrt(2000) * a few stages
TOL = {"fp64": 1e-13, "fp32": 2e-5}


@pytest.mark.parametrize("prec", ["fp64", "fp32"])
@pytest.mark.parametrize("Dl,Dr", [(1, 1), (3, 7), (8, 9), (16, 15), (17, 33), (31, 64),
                                   (65, 32), (129, 63), (128, 257), (400, 130)])
def test_heff_over_tile_edges(prec, Dl, Dr):
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
    ctx.close()
