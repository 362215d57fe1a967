"""The work that a user of this library has it do, as a list of measurable calls.

Every case goes through the public binding (paper_2505_23429_gb300).  The operators are the
library's own workloads: the Heisenberg chain with L = 12 sites and the random chemistry
Hamiltonian with L = 8, 12 or 16 orbitals (seeds and bond dimensions of synthetic.configs),
whose MPO bond dimension reaches 562 at L = 16.  Tensors that a sweep would hand over
(environments, two-site vectors, cores) are drawn from the seed with the symmetries and the
spread of magnitudes that they have there.
"""
import functools
import math

import numpy as np
import torch

import paper_2505_23429_gb300 as a2
from synthetic import chemistry_integrals, chemistry_mpo, heisenberg_mpo

SEED_INT = 2505          # integrals of the chemistry workloads
SINGLE = ("bf16", "f32emu", "fp32")   # results are single precision (or less)


def listed():
    return [
        # the smallest call: one FP64 operator application of the Heisenberg workload, all
        # launches and latency
        dict(name="heff_fp64_heisenberg_D32", op="heff", model="heisenberg", L=12, k=5, Dl=32,
             Dr=32, prec="fp64"),
        # the tensor-core Lanczos phases at a middle bond of the L = 16 workload, D = 256
        dict(name="heff_bf16_chem_D256", op="heff", model="chemistry", L=16, k=5, Dl=256,
             Dr=256, prec="bf16"),
        # ... and its FP32-accurate products at the bond of the hand-over core, the densest
        dict(name="heff_f32emu_chem_D256_handover", op="heff", model="chemistry", L=16, k=7,
             Dl=256, Dr=256, prec="f32emu"),
        # the FP64 refinement of a Ritz pair: one FP64-class application per local problem
        dict(name="heff_f64emu_chem_D256", op="heff", model="chemistry", L=16, k=5, Dl=256,
             Dr=256, prec="f64emu"),
        # environment updates, the most frequent step of an iteration: full size, left
        dict(name="env_left_f64emu_chem_D256", op="env", model="chemistry", L=16, j=5, side=0,
             Dlb=256, Drb=256, Dlk=256, Drk=256, prec="f64emu"),
        # ... and right, bra and ket of different odd bond dimensions (a coarse cross entry)
        dict(name="env_right_f64emu_chem_ragged", op="env", model="chemistry", L=12, j=7, side=1,
             Dlb=93, Drb=121, Dlk=87, Drk=110, prec="f64emu"),
        # truncated SVD of a two-site tensor after a local solve
        dict(name="svd_two_site_D256", op="svd", Dl=256, n1=4, n2=4, Dr=256, D_max=256),
        # truncated SVD inside the TT rounding (a core against the summed bond), odd sizes
        dict(name="svd_rounding_ragged", op="svd", Dl=199, n1=4, n2=1, Dr=597, D_max=199),
        # LQ inside the TT rounding: the summed bond against a core, odd sizes
        dict(name="lq_rounding_ragged", op="lq", rows=597, cols=2388),
        # whole call: one global iteration, FP64, groups on concurrent streams
        dict(name="sweep_fp64_heisenberg_D32", op="sweep", model="heisenberg", L=12, D=32, P=2,
             prec="fp64", tol=1e-10, sequential=False),
        # whole call: one global iteration in mixed precision with the FP64 refinement
        dict(name="sweep_mixed_chem_D64", op="sweep", model="chemistry", L=8, D=64, P=2,
             prec="bf16", tol=1e-6, sequential=True),
        # the backward direction: the energy's gradient with respect to all integrals
        dict(name="gradient_chem_D64", op="gradient", L=8, D=64),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    op = rng.choice(["heff", "heff", "heff", "env", "env", "svd", "lq", "sweep", "gradient"])
    if op in ("heff", "env"):
        model = rng.choice(["heisenberg", "chemistry", "chemistry", "chemistry"])
        L = 12 if model == "heisenberg" else rng.choice([8, 12, 16])
        prec = rng.choice(["fp64", "fp32", "bf16", "f32emu", "f64emu", "f64emu"])
        # the FP64 and FP32 operators are used on small problems
        top = 64 if model == "heisenberg" else 96 if prec in ("fp64", "fp32") else 256
        low = 8 if prec in ("fp64", "fp32") or model == "heisenberg" else 24
        if op == "heff":
            if prec == "f64emu":
                top = min(top, 200)
            return dict(op="heff", model=model, L=L, k=rng.randint(1, L - 3),
                        Dl=_log_int(rng, low, top), Dr=_log_int(rng, low, top), prec=prec)
        return dict(op="env", model=model, L=L, j=rng.randint(1, L - 2), side=rng.randint(0, 1),
                    Dlb=_log_int(rng, low, top), Drb=_log_int(rng, low, top),
                    Dlk=_log_int(rng, low, top), Drk=_log_int(rng, low, top), prec=prec)
    if op == "svd":
        Dl, Dr = _log_int(rng, 4, 256), _log_int(rng, 4, 256)
        n1, n2 = rng.choice([(2, 2), (4, 4), (4, 1), (4, 4)])
        if n2 == 1:
            Dr = min(3 * Dr, 768)
        return dict(op="svd", Dl=Dl, n1=n1, n2=n2, Dr=Dr,
                    D_max=max(1, min(256, min(Dl * n1, n2 * Dr) * rng.randint(1, 4) // 4)))
    if op == "lq":
        Dl = _log_int(rng, 8, 640)
        return dict(op="lq", rows=Dl, cols=max(2, int(Dl * rng.uniform(0.5, 4.0))))
    if op == "sweep":
        if rng.random() < 0.5:
            return dict(op="sweep", model="heisenberg", L=rng.randint(8, 12),
                        D=_log_int(rng, 8, 32), P=rng.randint(1, 3), prec="fp64", tol=1e-10,
                        sequential=rng.random() < 0.5)
        return dict(op="sweep", model="chemistry", L=rng.choice([6, 8]), D=_log_int(rng, 16, 64),
                    P=rng.randint(1, 3), prec=rng.choice(["bf16", "f32emu"]), tol=1e-6,
                    sequential=rng.random() < 0.5)
    return dict(op="gradient", L=rng.choice([6, 8]), D=_log_int(rng, 12, 64))


# ------------------------------------------------------------------ what a program keeps
@functools.lru_cache(maxsize=None)
def _context():
    st = torch.cuda.Stream()
    return st, a2.Context(0, stream=st.cuda_stream)


@functools.lru_cache(maxsize=None)
def _host_mpo(model, L, coeff_map=False):
    if model == "heisenberg":
        return heisenberg_mpo(L)
    h, eri = chemistry_integrals(L, SEED_INT)
    return chemistry_mpo(h, eri, coeff_map=coeff_map)


@functools.lru_cache(maxsize=None)
def _mpo(model, L):
    return a2.MPO(_context()[1], _host_mpo(model, L))


def _gen(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(int(seed))
    return g


def _randn(g, *shape):
    return torch.randn(*shape, generator=g, dtype=torch.float64, device="cuda")


def _environment(g, bra, R, ket):
    """[bra][MPO bond][ket]: entries ~ 1/sqrt(D), the MPO channels spread over two decades,
    symmetric in (bra, ket) where the two dimensions agree."""
    e = _randn(g, bra, R, ket) / math.sqrt(max(bra, ket))
    u = torch.rand(R, generator=g, dtype=torch.float64, device="cuda")
    e *= (10.0 ** (-2.0 * u))[None, :, None]
    return (0.5 * (e + e.permute(2, 1, 0))).contiguous() if bra == ket else e


def _orthonormal(g, rows, cols):
    q, _ = torch.linalg.qr(_randn(g, max(rows, cols), min(rows, cols)))
    return q if rows >= cols else q.T.contiguous()


def _bonds(n, L, D):
    return [int(min(D, n ** min(j, L - j, 40))) for j in range(L + 1)]


def _random_tt(n, L, D, seed):
    """Left-orthogonal unit-norm cores of full bond dimension (host, FP64)."""
    rng = np.random.default_rng(int(seed))
    b = _bonds(n, L, D)
    cores = []
    for j in range(L):
        q, _ = np.linalg.qr(rng.standard_normal((b[j] * n, b[j + 1])))
        cores.append(np.ascontiguousarray(q.reshape(b[j], n, b[j + 1])))
    cores[-1] /= np.linalg.norm(cores[-1])
    return cores


def _heff_inputs(case, seed, W1, W2):
    g = _gen(seed)
    Dl, Dr = case["Dl"], case["Dr"]
    Lenv = _environment(g, Dl, W1.shape[0], Dl)
    Renv = _environment(g, Dr, W2.shape[3], Dr)
    x = _randn(g, Dl, W1.shape[1], W2.shape[1], Dr)
    return Lenv, Renv, x / x.norm()


def _env_inputs(case, seed, W):
    g = _gen(seed)
    n = W.shape[1]
    Dlb, Drb, Dlk, Drk = (case[k] for k in ("Dlb", "Drb", "Dlk", "Drk"))
    if case["side"] == 0:
        Hin = _environment(g, Dlb, W.shape[0], Dlk)
        bra = _orthonormal(g, Dlb * n, Drb).reshape(Dlb, n, Drb)
        ket = bra if (Dlb, Drb) == (Dlk, Drk) else \
            _orthonormal(g, Dlk * n, Drk).reshape(Dlk, n, Drk)
    else:
        Hin = _environment(g, Drb, W.shape[3], Drk)
        bra = _orthonormal(g, Dlb, n * Drb).reshape(Dlb, n, Drb)
        ket = bra if (Dlb, Drb) == (Dlk, Drk) else \
            _orthonormal(g, Dlk, n * Drk).reshape(Dlk, n, Drk)
    return Hin, bra.contiguous(), ket.contiguous()


def _svd_input(case, seed):
    """Two-site tensor with slowly decaying, distinct Schmidt values."""
    g = _gen(seed)
    rows, cols = case["Dl"] * case["n1"], case["n2"] * case["Dr"]
    n = min(rows, cols)
    s = (1.0 + torch.arange(n, dtype=torch.float64, device="cuda") / 20.0) ** -1.5
    x = (_orthonormal(g, rows, n) * (s / s.norm())) @ _orthonormal(g, n, cols)
    return x.reshape(case["Dl"], case["n1"], case["n2"], case["Dr"]).contiguous()


def _lq_input(case, seed):
    """Rows of graded norms, as the weighted sum of tensor trains has them."""
    g = _gen(seed)
    m = _randn(g, case["rows"], case["cols"]) / math.sqrt(case["cols"])
    u = torch.rand(case["rows"], generator=g, dtype=torch.float64, device="cuda")
    return (m * (10.0 ** (-3.0 * u))[:, None]).contiguous()


def prepare(case, seed):
    st, ctx = _context()
    op = case["op"]
    new = functools.partial(torch.zeros, dtype=torch.float64, device="cuda")
    s = dict(case=case, ctx=ctx, stream=st)
    if op == "heff":
        W = _host_mpo(case["model"], case["L"])
        k = case["k"]
        Lenv, Renv, x = _heff_inputs(case, seed, W[k], W[k + 1])
        torch.cuda.synchronize()
        s.update(x=x, y=torch.zeros_like(x), op=a2.HeffOp(
            ctx, _mpo(case["model"], case["L"]), k, Lenv, Renv, prec=case["prec"]))
    elif op == "env":
        W = _host_mpo(case["model"], case["L"])[case["j"]]
        Hin, bra, ket = _env_inputs(case, seed, W)
        shape = (case["Drb"], W.shape[3], case["Drk"]) if case["side"] == 0 else \
            (case["Dlb"], W.shape[0], case["Dlk"])
        s.update(mpo=_mpo(case["model"], case["L"]), Hin=Hin, bra=bra, ket=ket, out=new(shape))
    elif op == "svd":
        rows, cols = case["Dl"] * case["n1"], case["n2"] * case["Dr"]
        n = min(rows, cols)
        s.update(x=_svd_input(case, seed), P=new(rows * n), SQ=new(n * cols))
    elif op == "lq":
        k = min(case["rows"], case["cols"])
        s.update(M=_lq_input(case, seed), Lo=new(case["rows"], k), Q=new(k, case["cols"]))
    elif op == "sweep":
        n = 2 if case["model"] == "heisenberg" else 4
        cores = _random_tt(n, case["L"], case["D"], seed)
        s.update(mpo=_mpo(case["model"], case["L"]), cores=cores, tt=a2.TT.from_cores(ctx, cores))
    else:
        W, cmap = _host_mpo("chemistry", case["L"], True)
        cores = _random_tt(4, case["L"], case["D"], seed)
        s.update(mpo=_mpo("chemistry", case["L"]), cmap=cmap, tt=a2.TT.from_cores(ctx, cores))
    torch.cuda.synchronize()
    return s


def _dense_state(cores):
    """The vector that the tensor train stands for: what the new state is up to the choice
    of basis on each bond, which the cores alone leave open."""
    v = np.ones((1, 1))
    for c in cores:
        v = (v @ c.reshape(c.shape[0], -1)).reshape(-1, c.shape[2])
    return v.ravel()


def _sign_fixed(P, SQ):
    """Singular vectors with the usual sign choice: each left vector's largest entry > 0."""
    sg = torch.gather(P, 0, P.abs().argmax(0, keepdim=True)).sign()
    return P * sg, SQ * sg.reshape(-1, 1)


def run(s):
    case, ctx = s["case"], s["ctx"]
    op = case["op"]
    with torch.cuda.stream(s["stream"]):
        if op == "heff":
            s["op"].apply(s["x"], s["y"])
            return s["y"].float() if case["prec"] in SINGLE else s["y"]
        if op == "env":
            a2.env_update(ctx, s["mpo"], case["j"], case["side"], s["Hin"], s["bra"], s["ket"],
                          s["out"], prec=case["prec"])
            return s["out"].float() if case["prec"] in SINGLE else s["out"]
        if op == "svd":
            r, disc = a2.svd_split(ctx, s["x"], case["D_max"], 1e-6, s["P"], s["SQ"])
            rows, cols = case["Dl"] * case["n1"], case["n2"] * case["Dr"]
            P, SQ = _sign_fixed(s["P"][:rows * r].view(rows, r), s["SQ"][:r * cols].view(r, cols))
            return dict(P=P, SQ=SQ, rank=r, discarded=disc)
        if op == "lq":
            a2.lq(ctx, s["M"], s["Lo"], s["Q"])
            return dict(L=s["Lo"], Q=s["Q"])
        if op == "sweep":
            for j, c in enumerate(s["cores"]):
                s["tt"].set_core(j, c)
            r = a2.additive_sweep(ctx, s["tt"], s["mpo"], case["P"], D_max=case["D"],
                                  svd_tol=case["tol"], eig_tol=case["tol"], prec=case["prec"],
                                  sequential=case["sequential"])
            return dict(energy_in=r["energy_in"], lambda_coarse=r["lambda_coarse"],
                        energy_local=r["energy_local"], S_hat=r["S_hat"], A_hat=r["A_hat"],
                        state=_dense_state(s["tt"].cores()))
        E, g = a2.energy_gradient(ctx, s["tt"], s["mpo"], s["cmap"])
        return dict(energy=E, grad=g)


# ------------------------------------------------------------------ the work of one pass
def _nnz(W):
    return float(np.count_nonzero(W))


def _heff_flops(W1, W2, Dl, Dr):
    n1, n2 = W1.shape[1], W2.shape[1]
    return 2.0 * n1 * n2 * Dl * Dr * (W1.shape[0] * Dl + W2.shape[3] * Dr) + \
        2.0 * Dl * Dr * (n2 * _nnz(W1) + n1 * _nnz(W2))


def _env_work(W, side, Dlb, Drb, Dlk, Drk):
    Rl, n, _, Rr = W.shape
    if side == 0:
        fl = 2.0 * n * (Dlb * Rl * Dlk * Drk + Drb * Rr * Dlb * Drk) + 2.0 * Dlb * Drk * _nnz(W)
    else:
        fl = 2.0 * n * (Drb * Rr * Drk * Dlk + Dlb * Rl * Drb * Dlk) + 2.0 * Drb * Dlk * _nnz(W)
    by = 8.0 * (Dlb * Rl * Dlk + Drb * Rr * Drk + n * (Dlb * Drb + Dlk * Drk))
    return by + 16.0 * _nnz(W), fl


def work(case):
    op = case["op"]
    if op == "heff":
        W = _host_mpo(case["model"], case["L"])
        W1, W2 = W[case["k"]], W[case["k"] + 1]
        Dl, Dr = case["Dl"], case["Dr"]
        size = {"fp64": 8, "f64emu": 8, "bf16": 2}.get(case["prec"], 4)   # environments
        return {"bytes": size * (Dl * Dl * W1.shape[0] + Dr * Dr * W2.shape[3]) +
                16.0 * (Dl * Dr * W1.shape[1] * W2.shape[1] + _nnz(W1) + _nnz(W2)),
                "flops": _heff_flops(W1, W2, Dl, Dr)}
    if op == "env":
        by, fl = _env_work(_host_mpo(case["model"], case["L"])[case["j"]], case["side"],
                           *(case[k] for k in ("Dlb", "Drb", "Dlk", "Drk")))
        return {"bytes": by, "flops": fl}
    if op == "svd":
        rows, cols = case["Dl"] * case["n1"], case["n2"] * case["Dr"]
        m, n = max(rows, cols), min(rows, cols)
        r = min(n, case["D_max"])
        return {"bytes": 8.0 * (rows * cols + r * (rows + cols)),
                "flops": 4.0 * m * n * n - 4.0 / 3.0 * n ** 3 + 4.0 * rows * n * r +
                2.0 * r * rows * cols}
    if op == "lq":
        r, c = case["rows"], case["cols"]
        k = min(r, c)
        return {"bytes": 8.0 * (r * c + r * k + k * c),
                "flops": 2.0 * (2.0 * r * c * k - (r + c) * k * k + 2.0 / 3.0 * k ** 3) +
                2.0 * k * k * c}
    if op == "sweep":   # one operator application per bond and the environments, at least
        n = 2 if case["model"] == "heisenberg" else 4
        W, b = _host_mpo(case["model"], case["L"]), _bonds(n, case["L"], case["D"])
        fl = sum(_heff_flops(W[k], W[k + 1], b[k], b[k + 2]) for k in range(case["L"] - 1))
        fl += 2 * sum(_env_work(W[j], 0, b[j], b[j + 1], b[j], b[j + 1])[1]
                      for j in range(case["L"]))
        by = sum(16.0 * b[j] * n * b[j + 1] + 16.0 * _nnz(W[j]) for j in range(case["L"]))
        return {"bytes": by, "flops": fl}
    W, cmap = _host_mpo("chemistry", case["L"], True)
    b = _bonds(4, case["L"], case["D"])
    # forward: one chain of updates; backward: the right environments and each core's adjoint
    fl = 4 * sum(_env_work(W[j], 0, b[j], b[j + 1], b[j], b[j + 1])[1] for j in range(case["L"]))
    by = sum(8.0 * b[j] * 4 * b[j + 1] + 16.0 * _nnz(W[j]) for j in range(case["L"]))
    return {"bytes": by + 28.0 * len(cmap["param"]) + 8.0 * cmap["nparam"], "flops": fl}


# ------------------------------------------------------------------ plain 64-bit results
def _dev(a):
    return torch.from_numpy(np.ascontiguousarray(a)).cuda()


def _left(E, bra, W, ket):
    """out[b,v,d] = sum bra[a,s,b] E[a,w,c] W[w,s,t,v] ket[c,t,d]"""
    t = torch.tensordot(E, ket, ([2], [0]))               # a w t d
    t = torch.tensordot(t, W, ([1, 2], [0, 2]))           # a d s v
    return torch.tensordot(bra, t, ([0, 1], [0, 2])).permute(0, 2, 1)   # b d v -> b v d


def _right(E, bra, W, ket):
    """out[a,w,c] = sum bra[a,s,b] W[w,s,t,v] E[b,v,d] ket[c,t,d]"""
    t = torch.tensordot(E, ket, ([2], [2]))               # b v c t
    t = torch.tensordot(t, W, ([1, 3], [3, 2]))           # b c w s
    return torch.tensordot(bra, t, ([1, 2], [3, 0])).permute(0, 2, 1)   # a c w -> a w c


def _energy(cores, W):
    E = torch.ones(1, 1, 1, dtype=torch.float64, device="cuda")
    N = torch.ones(1, 1, dtype=torch.float64, device="cuda")
    for c, w in zip(cores, W):
        E = _left(E, c, w, c)
        N = torch.tensordot(c, torch.tensordot(N, c, ([1], [0])), ([0, 1], [0, 1]))
    return E.reshape(()) / N.reshape(())


def exact(case, seed):
    op = case["op"]
    if op == "heff":
        Wh = _host_mpo(case["model"], case["L"])
        W1, W2 = _dev(Wh[case["k"]]), _dev(Wh[case["k"] + 1])
        Lenv, Renv, x = _heff_inputs(case, seed, W1, W2)
        t = torch.tensordot(Lenv, x, ([2], [0]))              # a w t1 t2 b
        t = torch.tensordot(t, W1, ([1, 2], [0, 2]))          # a t2 b s1 v
        t = torch.tensordot(t, W2, ([4, 1], [0, 2]))          # a b s1 s2 u
        return torch.tensordot(t, Renv, ([4, 1], [1, 2])).contiguous()   # a s1 s2 b
    if op == "env":
        W = _dev(_host_mpo(case["model"], case["L"])[case["j"]])
        Hin, bra, ket = _env_inputs(case, seed, W)
        return (_left if case["side"] == 0 else _right)(Hin, bra, W, ket).contiguous()
    if op == "svd":
        x = _svd_input(case, seed)
        M = x.reshape(case["Dl"] * case["n1"], -1).cpu()
        U, s, Vh = torch.linalg.svd(M, full_matrices=False)
        tail = torch.sqrt(torch.flip(torch.cumsum(torch.flip(s * s, [0]), 0), [0]))
        fit = [k for k in range(1, len(s) + 1)
               if (float(tail[k]) if k < len(s) else 0.0) <= 1e-6 * float(tail[0])]
        r = max(1, min(fit[0], case["D_max"]))
        P, SQ = _sign_fixed(U[:, :r], s[:r, None] * Vh[:r])
        return dict(P=P, SQ=SQ, rank=r, discarded=float(tail[r]) if r < len(s) else 0.0)
    if op == "lq":
        q, r = torch.linalg.qr(_lq_input(case, seed).cpu().T)
        sg = torch.where(torch.diagonal(r) < 0, -1.0, 1.0).to(torch.float64)
        return dict(L=(r.T * sg).contiguous(), Q=(q * sg).T.contiguous())
    if op == "sweep":   # the iterate's Rayleigh quotient; the rest depends on the solvers' stops
        n = 2 if case["model"] == "heisenberg" else 4
        cores = [_dev(c) for c in _random_tt(n, case["L"], case["D"], seed)]
        E = float(_energy(cores, [_dev(w) for w in _host_mpo(case["model"], case["L"])]))
        return dict(energy_in=E, lambda_coarse=None, energy_local=None, S_hat=None, A_hat=None,
                    state=None)
    W, cmap = _host_mpo("chemistry", case["L"], True)
    Wd = [_dev(w).requires_grad_() for w in W]
    cores = [_dev(c) for c in _random_tt(4, case["L"], case["D"], seed)]
    E = _energy(cores, Wd)
    dW = torch.autograd.grad(E, Wd)
    g = np.zeros(int(cmap["nparam"]))
    for j, d in enumerate(dW):
        at = cmap["site"] == j
        np.add.at(g, cmap["param"][at], d.reshape(-1).cpu().numpy()[cmap["index"][at]] *
                  cmap["factor"][at])
    return dict(energy=float(E.detach()), grad=g)
