"""The energy's derivative with respect to single MPO elements: every element of every core,
and maps of a few elements named several times, at bond dimensions below and around a warp,
against NumPy."""
import numpy as np
import pytest

from oracle.env import left_envs, right_envs
from synthetic import heisenberg_mpo, random_tt_cores

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

import paper_2505_23429_gb300 as a2  # noqa: E402

# sums of at most 4 * 37^2 products of FP64 rounding, relative to the largest derivative
TOL = 1e-12


@pytest.mark.parametrize("few", [False, True])
@pytest.mark.parametrize("L,D", [(2, 2), (5, 3), (10, 32), (12, 37)])
def test_elements(few, L, D):
    m = heisenberg_mpo(L)
    cores = random_tt_cores([2] * L, D, 7)
    HL, HR = left_envs(cores, m), right_envs(cores, m)
    n2 = np.ones((1, 1))
    for U in cores:
        n2 = np.einsum("ac,asb,csd->bd", n2, U, U, optimize=True)
    G = [np.einsum("awc,asb,ctd,bvd->wstv", HL[j], cores[j], cores[j], HR[j + 1],
                   optimize=True) / n2[0, 0] for j in range(L)]
    rng = np.random.default_rng(L)
    if few:
        site = rng.integers(0, L, 40)
        site[site == 1] = 0                         # one core without entries
        index = np.array([rng.integers(0, min(G[j].size, 9)) for j in site])
        param = rng.integers(0, 6, 40)
    else:
        site = np.concatenate([np.full(g.size, j) for j, g in enumerate(G)])
        index = np.concatenate([np.arange(g.size) for g in G])
        param = np.arange(len(site))
    factor = rng.standard_normal(len(site))
    ref = np.zeros(param.max() + 1)
    np.add.at(ref, param, factor * np.array([G[j].ravel()[i] for j, i in zip(site, index)]))
    ctx = a2.Context(0)
    tt = a2.TT.from_cores(ctx, cores)
    E, g = a2.energy_gradient(ctx, tt, a2.MPO(ctx, m), dict(
        param=param, site=site, index=index, factor=factor, nparam=len(ref)))
    assert np.abs(g - ref).max() < TOL * max(np.abs(ref).max(), max(np.abs(x).max() for x in G))
    E0 = np.sum(G[0] * m[0])
    assert abs(E - E0) < TOL * max(1.0, abs(E0), np.abs(G[0]).max())
    ctx.close()
