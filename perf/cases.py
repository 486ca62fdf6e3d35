"""What is timed: the calls that a program using this library makes, over the
sizes that it makes them at.

Six kinds of call:

* ``iterate``: one CTMRG iteration (ctm_converge with one iteration: the four
  directional moves over the whole cell and the corner-spectrum measure) from
  a context that has left its random start, then the corner spectra and one
  two-site density matrix. This is the work of a solve; it is timed in the
  default FP64 arithmetic, in the split bf16 x3 mode, and in the
  fp64-accurate exact-digit mode (split_refine = +inf).
* ``apply``: one enlarged corner and its product with an N x k block
  (ctm_corner_apply), the block that the subspace iteration is built of.
* ``energy``: the two-site density matrices of every bond of the cell
  (ctm_rdm2), as an optimisation evaluates them on an environment.
* ``gradient``: dE/dA through one recorded iteration (ctm_grad), the backward
  direction of the path.
* ``svdvals``: ctm_svdvals_noalloc on a matrix in device memory, the smallest
  call of the library.

What an iteration returns is what the environment fixes: corner spectra and
density matrices. Its corners and edges are fixed only up to rotations inside
nearly degenerate singular spaces, so they are not compared element by
element. A split-precision context computes its products to 24 bits and the
error of one product travels through all that follow, so a program that runs
whole iterations in that mode keeps their results in single precision; single
layers of it (``apply``) are returned as they come.
"""
import math

import numpy as np
import torch

import paper_2607_15158_gb300 as ctm

PHYS = 2            # physical dimension of every workload of this repository
OVERSAMPLING = 5    # p, k = chi + p
PRECISION = {"fp64": ctm.CTM_PREC_FP64, "split": ctm.CTM_PREC_SPLIT_BF16,
             "exact": ctm.CTM_PREC_SPLIT_BF16}
HEISENBERG = 0.25 * np.array([[1.0, 0, 0, 0], [0, -1.0, 2.0, 0], [0, 2.0, -1.0, 0], [0, 0, 0, 1.0]])


def _iterate(name, Lx, Ly, D, chi, cplx, prec, rounds=1, warm=6):
    return dict(name=name, kind="iterate", Lx=Lx, Ly=Ly, D=D, chi=chi, cplx=cplx, prec=prec,
                rounds=rounds, warm=warm)


def listed():
    return [
        # the singular values of one small device matrix: a program that owns
        # all device memory asks for a corner's spectrum
        dict(name="svdvals_f64_64", kind="svdvals", k=64, cplx=False),
        # the smallest solves, where launches and latency count: a first look
        # at a small bond dimension, and the candidates of a serving mix
        _iterate("iter_f64_1x1_D2_chi8", 1, 1, 2, 8, False, "fp64", rounds=2, warm=12),
        _iterate("iter_c128_3x3_D2_chi9", 3, 3, 2, 9, True, "fp64", warm=12),
        # the small workload of the benchmark suite (two rounds per projector)
        _iterate("iter_f64_1x1_D3_chi27", 1, 1, 3, 27, False, "fp64", rounds=2, warm=12),
        # ordinary solves in the default arithmetic: a complex cell with odd
        # block sizes, and the 3x3 D = 4 workload
        _iterate("iter_c128_2x2_D3_chi33", 2, 2, 3, 33, True, "fp64"),
        _iterate("iter_f64_3x3_D4_chi64", 3, 3, 4, 64, False, "fp64", warm=4),
        # fp64-accurate solves on the tensor cores
        _iterate("iter_exact_c128_2x2_D4_chi64", 2, 2, 4, 64, True, "exact", warm=4),
        # the benchmark's workload: split precision, 3x3 complex D = 6, chi = 144
        _iterate("iter_split_c128_3x3_D6_chi144", 3, 3, 6, 144, True, "split", warm=2),
        # an enlarged corner and its product with a block, in the two
        # arithmetics (the D = 6 workload for counters; odd sizes)
        dict(name="apply_split_c128_D6_chi80", kind="apply", D=6, chi=80, cplx=True, prec="split",
             herm=False),
        dict(name="apply_f64_D5_chi61_herm", kind="apply", D=5, chi=61, cplx=False, prec="fp64",
             herm=True),
        # the energy of a converged environment
        dict(name="energy_f64_2x2_D4_chi48", kind="energy", Lx=2, Ly=2, D=4, chi=48, cplx=False,
             prec="fp64"),
        # one gradient of an optimisation
        dict(name="grad_f64_1x1_D3_chi27", kind="gradient", D=3, chi=27, warm=8),
    ]


# ------------------------------------------------------------------- drawing
def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


# multiply-add budgets of a drawn iteration: those of the largest listed one
# of its arithmetic
_BUDGET = {"fp64": (3, 3, 4, 64, False, 1), "exact": (2, 2, 4, 64, True, 1),
           "split": (3, 3, 6, 144, True, 1)}


def draw(rng):
    kind = rng.choice(["iterate"] * 7 + ["apply"] * 2 + ["energy", "gradient", "svdvals"])
    if kind == "svdvals":
        return dict(kind=kind, k=_log_int(rng, 8, 128), cplx=rng.random() < 0.5)
    if kind == "gradient":
        D = rng.choice([2, 3])
        return dict(kind=kind, D=D, chi=_log_int(rng, 2 * D, 9 * D), warm=8)
    if kind == "energy":
        D = rng.choice([2, 3, 4])
        L = rng.choice([(1, 1), (2, 1), (2, 2)])
        return dict(kind=kind, Lx=L[0], Ly=L[1], D=D, chi=_log_int(rng, 2 * D, 12 * D),
                    cplx=rng.random() < 0.4, prec="fp64")
    if kind == "apply":
        prec = rng.choice(["fp64", "split"])
        D = rng.choice([3, 4, 5] if prec == "fp64" else [4, 5, 6, 7])
        top = 1500 if prec == "fp64" else 2880
        return dict(kind=kind, D=D, chi=_log_int(rng, 2 * D, top // (D * D)),
                    cplx=rng.random() < 0.5, prec=prec, herm=rng.random() < 0.5)
    prec = rng.choice(["fp64"] * 4 + ["split"] * 2 + ["exact"])
    budget = _macs_iteration(*_BUDGET[prec])
    while True:
        L = rng.choice([(1, 1), (2, 1), (1, 2), (2, 2), (3, 2), (3, 3)])
        D = rng.choice({"fp64": [2, 3, 4, 5], "split": [4, 5, 6], "exact": [3, 4, 5]}[prec])
        # the serving mix asks for chi between D^2 and 4 D^2
        chi = _log_int(rng, D * D, 4 * D * D)
        cplx, rounds = rng.random() < 0.5, rng.choice([1, 1, 2])
        if _macs_iteration(L[0], L[1], D, chi, cplx, rounds) <= budget:
            return dict(kind=kind, Lx=L[0], Ly=L[1], D=D, chi=chi, cplx=cplx, prec=prec,
                        rounds=rounds, warm=4)


# ------------------------------------------------------------------ the work
def _corner_macs(D, chi):
    """Multiply-adds of one enlarged corner: C T, (C T) T, A and conj(A)."""
    return chi**3 * D**2 + chi**3 * D**4 + 2 * chi**2 * PHYS * D**6


def _macs_iteration(Lx, Ly, D, chi, cplx, rounds):
    """Real multiply-adds of one iteration: per cut four corners, the corner
    products of the rounds and the half systems, rho and the absorption."""
    N = chi * D * D
    k = min(chi + OVERSAMPLING, N)
    cut = (4 * _corner_macs(D, chi) + (16 * rounds + 4) * N * N * k + N * k * k
           + chi**3 * D**2 + 2 * chi**3 * D**4 + 2 * chi**2 * PHYS * D**6)
    return 4 * Lx * Ly * cut * (4 if cplx else 1)


def work(case):
    es = 16 if case.get("cplx") else 8
    mul = 8 if case.get("cplx") else 2
    if case["kind"] == "svdvals":
        k = case["k"]
        # a bidiagonalisation, 8/3 k^3 flops, and the values from it
        return {"bytes": es * k * k + 8 * k, "flops": 4 * mul / 3 * k**3}
    D, chi = case["D"], case["chi"]
    N = chi * D * D
    k = min(chi + OVERSAMPLING, N)
    site = chi * chi * (1 + D * D)
    if case["kind"] == "iterate":
        S = case["Lx"] * case["Ly"]
        state = 4 * S * (site + 2 * N * k)   # C, T, X, W: read and written once
        return {"bytes": 2 * es * state,
                "flops": 2 * _macs_iteration(case["Lx"], case["Ly"], D, chi, case["cplx"],
                                             case["rounds"])}
    if case["kind"] == "apply":
        return {"bytes": es * (chi * chi * (1 + 2 * D * D) + 2 * PHYS * D**4 + 2 * N * k),
                "flops": mul * (_corner_macs(D, chi) + N * N * k)}
    half = _corner_macs(D, chi) + 2 * chi**3 * PHYS**2 * D**4   # half a two-site patch
    if case["kind"] == "energy":
        S = case["Lx"] * case["Ly"]
        return {"bytes": es * 4 * S * site, "flops": mul * 2 * S * (2 * half + chi**2 * 16 * D * D)}
    # gradient: the recorded iteration again, then about twice its work backward
    return {"bytes": es * (4 * site + 8 * N * k + PHYS * D**4),
            "flops": 2 * 3 * _macs_iteration(1, 1, D, chi, False, 1) + mul * 4 * half}


# ------------------------------------------------------------------- inputs
def _normal(rng, shape, cplx):
    x = rng.standard_normal(shape)
    return (x + 1j * rng.standard_normal(shape)) / math.sqrt(2.0) if cplx else x


def _tensors(rng, S, D, cplx):
    """One random on-site tensor A[s, u, l, d, r] of unit norm per site."""
    out = []
    for _ in range(S):
        A = _normal(rng, (PHYS, D, D, D, D), cplx)
        out.append(A / np.linalg.norm(A))
    return out


def _environment(rng, S, D, chi, cplx):
    """Corners and edges of the form a converged environment has: decaying
    corner spectra, edges that join equal bonds and like ket and bra legs,
    both with a random part."""
    w = np.diag(np.exp(-4.0 * np.arange(chi) / chi))
    C = np.empty((4, S, chi, chi), complex if cplx else float)
    T = np.empty((4, S, chi, chi, D, D), C.dtype)
    for i in range(4):
        for s in range(S):
            C[i, s] = w + 0.2 * _normal(rng, (chi, chi), cplx) / chi
            T[i, s] = (np.einsum("ab,uv->abuv", np.eye(chi), np.eye(D))
                       + 0.2 * _normal(rng, (chi, chi, D, D), cplx) / math.sqrt(chi))
            C[i, s] /= np.linalg.norm(C[i, s])
            T[i, s] /= np.linalg.norm(T[i, s])
    return C, T


def _inputs(case, seed):
    """The tensors, environment and block of an apply or energy case."""
    rng = np.random.default_rng(seed)
    S = case.get("Lx", 1) * case.get("Ly", 1)
    D, chi, cplx = case["D"], case["chi"], case["cplx"]
    A = _tensors(rng, S, D, cplx)
    C, T = _environment(rng, S, D, chi, cplx)
    N = chi * D * D
    Z = _normal(rng, (N, min(chi + OVERSAMPLING, N)), cplx) if case["kind"] == "apply" else None
    return A, C, T, Z


def _matrix(case, seed):
    """The k x k matrix of svdvals: a corner with a decaying spectrum."""
    g = torch.Generator(device="cuda").manual_seed(seed)
    k, t = case["k"], torch.complex128 if case["cplx"] else torch.float64
    M = torch.randn(k, k, dtype=t, device="cuda", generator=g)
    scale = torch.exp(-8.0 * torch.arange(k, device="cuda", dtype=torch.float64) / k)
    return M * scale[:, None] * scale[None, :]


def _options(case, seed):
    o = ctm.ctm_default_opts(p=OVERSAMPLING, seed=seed, prec=PRECISION[case.get("prec", "fp64")],
                             si_rounds=case.get("rounds", 1), warmup_iters=1, warmup_rounds=3)
    if case.get("prec") == "exact":
        o.split_refine = math.inf
    return o


def prepare(case, seed):
    if case["kind"] == "svdvals":
        return dict(case=case, A=_matrix(case, seed),
                    s=torch.empty(case["k"], dtype=torch.float64, device="cuda"))
    D, chi, cplx = case["D"], case["chi"], case.get("cplx", False)
    Lx, Ly = case.get("Lx", 1), case.get("Ly", 1)
    if case["kind"] in ("apply", "energy"):
        A, C, T, Z = _inputs(case, seed)
        ctx = ctm.ctm_init(Lx, Ly, A, PHYS, D, chi, cplx=cplx, opts=_options(case, seed))
        ctx.ctm_set_env(C, T)
        return dict(case=case, ctx=ctx, Z=Z)
    A = _tensors(np.random.default_rng(seed), Lx * Ly, D, cplx)
    ctx = ctm.ctm_init(Lx, Ly, A, PHYS, D, chi, cplx=cplx, opts=_options(case, seed))
    ctx.ctm_converge(0.0, case["warm"])
    if case["kind"] == "gradient":
        ctx.ctm_record(True)
        ctx.ctm_converge(0.0, 1)
        ctx.ctm_record(False)
    return dict(case=case, ctx=ctx)


def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "svdvals":
        ctm.ctm_svdvals_noalloc(state["A"].data_ptr(), case["k"],
                                ctm.CTM_C128 if case["cplx"] else ctm.CTM_F64,
                                state["s"].data_ptr(), torch.cuda.current_stream().cuda_stream)
        return state["s"]
    ctx = state["ctx"]
    if kind == "apply":
        return ctx.ctm_corner_apply(0, 0, 0, 1, state["Z"], herm=case["herm"])
    if kind == "energy":
        return [ctx.ctm_rdm2(x, y, d) for y in range(case["Ly"]) for x in range(case["Lx"])
                for d in (0, 1)]
    if kind == "gradient":
        E, dA = ctx.ctm_grad(HEISENBERG)
        return {"E": E, "dA": dA}
    ctx.ctm_converge(0.0, 1)
    s, rho = ctx.ctm_spectra(), ctx.ctm_rdm2(0, 0, 0)
    if case["prec"] == "split":
        return {"spectra": s.astype(np.float32), "rho": rho.astype(np.complex64)}
    return {"spectra": s, "rho": rho}


# ----------------------------------------------------------- 64-bit results
def _dev(x):
    return torch.from_numpy(np.ascontiguousarray(x)).cuda()


def _exact_corner(A, C, T):
    """The upper-left enlarged corner of a 1 x 1 cell as an N x N matrix."""
    a, c, t1, t4 = _dev(A[0]), _dev(C[0, 0]), _dev(T[0, 0]), _dev(T[3, 0])
    chi, D = c.shape[0], a.shape[1]
    x = torch.einsum("pm,mnuv->pnuv", c, t1)
    x = torch.einsum("tplw,pnuv->tlwnuv", t4, x)
    x = torch.einsum("tlwnuv,sulde->twnvsde", x, a)
    x = torch.einsum("twnvsde,svwDE->tdDneE", x, a.conj())
    return x.reshape(chi * D * D, chi * D * D)


def _exact_rdm(case, A, C, T, x, y, direction):
    """Density matrix of the bond from (x, y) to its right or lower neighbour;
    a vertical bond is a horizontal one of the cell turned by a quarter."""
    Lx, Ly = case["Lx"], case["Ly"]
    if direction == 0:
        s1, s2 = y * Lx + x, y * Lx + (x + 1) % Lx
        turn = 0
    else:
        s1, s2 = y * Lx + x, ((y + 1) % Ly) * Lx + x
        turn = 1

    def c(i, s):
        return _dev(C[(i + turn) % 4, s])

    def t(i, s):
        return _dev(T[(i + turn) % 4, s])

    def ket(s):
        a = _dev(A[s])
        return a.permute(0, 4, 1, 2, 3) if turn else a

    k1, k2 = ket(s1), ket(s2)
    e = torch.einsum
    L = e("ab,bcuU->acuU", c(0, s1), t(0, s1))
    L = e("kalL,acuU->klLcuU", t(3, s1), L)
    L = e("klLcuU,sulxm->kLcUsxm", L, k1)
    L = e("kLcUsxm,tULXM->kcsxmtXM", L, k1.conj())
    L = e("kcsxmtXM,jk->jcsxmtXM", L, c(3, s1))
    L = e("jcsxmtXM,ijxX->icsmtM", L, t(2, s1))
    R = e("ceoO,ef->cfoO", t(0, s2), c(1, s2))
    R = e("cfoO,fgrR->cgoOrR", R, t(1, s2))
    R = e("cgoOrR,qomwr->cgORqmw", R, k2)
    R = e("cgORqmw,vOMWR->cgqmwvMW", R, k2.conj())
    R = e("cgqmwvMW,gh->chqmwvMW", R, c(2, s2))
    R = e("chqmwvMW,hiwW->ciqmvM", R, t(2, s2))
    rho = e("icsmtM,ciqmvM->sqtv", L, R).reshape(PHYS**2, PHYS**2)
    rho = rho / torch.trace(rho)
    return rho.to(torch.complex128).cpu().numpy()


def exact(case, seed):
    if case["kind"] == "svdvals":
        return torch.linalg.svdvals(_matrix(case, seed))
    if case["kind"] == "apply":
        A, C, T, Z = _inputs(case, seed)
        Q = _exact_corner(A, C, T)
        return ((Q.conj().T if case["herm"] else Q) @ _dev(Z)).cpu().numpy()
    if case["kind"] == "energy":
        A, C, T, _ = _inputs(case, seed)
        return [_exact_rdm(case, A, C, T, x, y, d) for y in range(case["Ly"])
                for x in range(case["Lx"]) for d in (0, 1)]
    # an iteration starts from the state that earlier ones left, and a
    # gradient from its record
    return None
