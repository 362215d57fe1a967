"""A reduction of more than 2^24 entries through the column slicing (65536 chunks and a ragged
one): an environment update whose ket bond is that long, against plain FP64 products."""
import pytest

from synthetic import heisenberg_mpo

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

import paper_2505_23429_gb300 as a2  # noqa: E402


@pytest.mark.parametrize("K", [65536 * 256 - 300, 65536 * 256 + 300])
def test_long_reduction(K):
    m = heisenberg_mpo(4)
    ctx = a2.Context(0)
    g = torch.Generator(device="cuda")
    g.manual_seed(K)
    kw = dict(generator=g, dtype=torch.float64, device="cuda")
    Hin = torch.randn(1, 1, K, **kw)
    bra = torch.randn(1, 2, 1, **kw)
    ket = torch.randn(K, 2, 1, **kw)
    ket[-400:] *= 1e3                                     # the last chunks count
    out = torch.zeros(1, m[0].shape[3], 1, dtype=torch.float64, device="cuda")
    torch.cuda.synchronize()
    a2.env_update(ctx, a2.MPO(ctx, m), 0, 0, Hin, bra, ket, out, prec="f64emu")
    ctx.synchronize()
    W = torch.from_numpy(m[0][0]).cuda()                  # s t w'
    x = Hin.reshape(1, K) @ ket.reshape(K, 2)             # 1 t
    mag = Hin.abs().reshape(1, K) @ ket.abs().reshape(K, 2)
    ref = torch.einsum("s,stw,t->w", bra.reshape(2), W, x.reshape(2))
    scale = torch.einsum("s,stw,t->w", bra.abs().reshape(2), W.abs(), mag.reshape(2)).max()
    # FP32 pairs: 2^-48 of the largest partial sum, sums over 4096 splits in their low parts
    assert float((out.reshape(-1) - ref).abs().max() / scale) < 2.0 ** -42
    ctx.close()
