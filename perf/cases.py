"""The measured work of this library: what a user's program has it do, through the public calls.

A case names one call (or the short sequence of calls a program makes) and its sizes:

    contraction   esmp2.virtual_contraction_noalloc: S slices of Nv x Nv, bf16 operands
    sigma         Handle.sigma on a kept handle: one application of the zeroth-order operator
    solve         Handle(...), solve, energy (and the solution): one excited state from its integrals
    batch         esmp2.batch_solve on host arrays: several states or molecules of uneven size
    gradient      Handle.grad on a solved handle: dE2/dF and dE2/d(ia|jb)
    training      esmp2_energy(...).backward(): the differentiable energy, forward and backward

Sizes run from No=6 Nv=30 to No=30 Nv=400 (the configurations of the tests and of bench.py) with
Nv = 5 to 14 No between them.  Inputs follow the recipe of the synthetic workloads: occupied
orbital energies U[-2, -0.3], virtual ones U[0.2, 3], off-diagonal Fock elements N(0, sigma_off),
integrals N(0, 1e-2) with their permutational symmetry, and one dominant singles coefficient.
"""
import math

import numpy as np
import torch

from paper_2003_12923_gb300 import esmp2
from paper_2003_12923_gb300.autograd import esmp2_energy

PRECISION = {"fp64": esmp2.FP64, "fp64_tc": esmp2.FP64_TC, "bf16": esmp2.MIXED_BF16, "tf32": esmp2.MIXED_TF32,
             "reduced": esmp2.REDUCED_MIXED}
NOALLOC_LIMIT = 64 << 20
WEIGHTS = (0.5, 1.0, 0.5, 0.5, 2.0)   # determinant inner product of the T, S, X, Y, Z blocks


# ------------------------------------------------------------------------------------ the cases
def listed():
    return [
        # the allocation-free contraction inside another framework's loop: latency counts
        {"name": "contraction 16x64", "kind": "contraction", "S": 16, "Nv": 64},
        # one operator application of the smallest configuration (No=6 Nv=30), the step of an
        # iterative method that a program writes itself: launches count
        {"name": "sigma fp64 6x30", "kind": "sigma", "No": 6, "Nv": 30, "precision": "fp64"},
        # the same at a ragged ordinary size, in float64 and on the tensor cores
        {"name": "sigma fp64 13x113", "kind": "sigma", "No": 13, "Nv": 113, "precision": "fp64"},
        {"name": "sigma fp64_tc 20x200", "kind": "sigma", "No": 20, "Nv": 200, "precision": "fp64_tc"},
        # a whole small state in plain float64 (the smallest configuration)
        {"name": "solve fp64 6x30", "kind": "solve", "No": 6, "Nv": 30, "precision": "fp64", "tol": 1e-10,
         "sigma_off": 1e-3, "shift": 0.0, "solution": True},
        # the mixed-precision solves at ordinary sizes: bf16 (the default form), tf32 at a ragged
        # size, the reduced-cost basis
        {"name": "solve bf16 20x200", "kind": "solve", "No": 20, "Nv": 200, "precision": "bf16", "tol": 1e-10,
         "sigma_off": 1e-3, "shift": 0.0, "solution": True},
        {"name": "solve tf32 11x131", "kind": "solve", "No": 11, "Nv": 131, "precision": "tf32", "tol": 1e-10,
         "sigma_off": 1e-3, "shift": 0.0, "solution": True},
        {"name": "solve reduced 16x160", "kind": "solve", "No": 16, "Nv": 160, "precision": "reduced", "tol": 1e-10,
         "sigma_off": 1e-3, "shift": 0.0, "solution": True},
        # the benchmark: a large state to 1e-8, of which a program keeps the energies
        {"name": "solve bf16 30x400", "kind": "solve", "No": 30, "Nv": 400, "precision": "bf16", "tol": 1e-8,
         "sigma_off": 1e-3, "shift": 0.0, "solution": False},
        # several uneven states from host arrays (the batch configuration's lower half)
        {"name": "batch bf16 6 of 8-14", "kind": "batch", "shapes": "8x71 14x160 9x121 12x131 10x90 13x106",
         "precision": "bf16", "tol": 1e-8, "concurrency": 3},
        # backward: the analytic gradient of a solved state, and the differentiable energy as a
        # training loop calls it
        {"name": "gradient 12x120", "kind": "gradient", "No": 12, "Nv": 120},
        {"name": "training fp64 8x80", "kind": "training", "No": 8, "Nv": 80, "precision": "fp64", "tol": 1e-10},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["contraction", "sigma", "sigma", "solve", "solve", "solve", "batch", "gradient", "training"])
    if kind == "contraction":
        while True:
            S, Nv = _log_int(rng, 4, 400), _log_int(rng, 24, 400)
            if (2 + 4) * (S + 1) * Nv * (Nv + 8) + 4096 <= NOALLOC_LIMIT:
                return {"kind": kind, "S": S, "Nv": Nv}
    if kind == "sigma":
        p = rng.choice(["fp64", "fp64_tc"])
        No = _log_int(rng, 5, 16 if p == "fp64" else 20)
        return {"kind": kind, "No": No, "Nv": min(200, int(round(No * rng.uniform(5, 14)))), "precision": p}
    if kind == "solve":
        p = rng.choice(["fp64", "bf16", "bf16", "tf32", "reduced"])
        No = _log_int(rng, 5, 10 if p == "fp64" else 24)
        off, shift = rng.choice([(1e-4, 0.0), (1e-3, 0.0), (1e-3, 0.0), (1e-2, 0.5)])
        return {"kind": kind, "No": No, "Nv": min(260, int(round(No * rng.uniform(5, 14)))), "precision": p,
                "tol": 1e-10, "sigma_off": off, "shift": shift, "solution": True}
    if kind == "batch":
        shapes = []
        for _ in range(rng.randint(3, 6)):
            No = rng.randint(8, 13)
            shapes.append("%dx%d" % (No, int(round(No * rng.uniform(8, 12)))))
        return {"kind": kind, "shapes": " ".join(shapes), "precision": rng.choice(["bf16", "reduced"]), "tol": 1e-8,
                "concurrency": rng.choice([2, 3])}
    No = _log_int(rng, 5, 12 if kind == "gradient" else 8)
    c = {"kind": kind, "No": No, "Nv": min(120 if kind == "gradient" else 80, int(round(No * rng.uniform(6, 11))))}
    return c if kind == "gradient" else dict(c, precision="fp64", tol=1e-10)


def _shapes(case):
    return [tuple(int(v) for v in s.split("x")) for s in case["shapes"].split()]


# ------------------------------------------------------------------------------------ the inputs
def _gen(seed, k=0):
    return torch.Generator(device="cuda").manual_seed(1000003 * (int(seed) % (1 << 40)) + k)


def _instance(No, Nv, seed, sigma_off=1e-3, sigma_eri=1e-2):
    """F, (ia|jb), (ij|ka), (ia|bc) and C of one synthetic state, float64 on the GPU."""
    g, f8 = _gen(seed), dict(dtype=torch.float64, device="cuda")
    N = No + Nv
    F = torch.randn(N, N, generator=g, **f8).mul_(sigma_off).triu_(1)
    F = F + F.T
    d = torch.rand(N, generator=g, **f8)
    d[:No] = d[:No] * 1.7 - 2.0
    d[No:] = d[No:] * 2.8 + 0.2
    F.diagonal().copy_(d)
    ovov = torch.randn(No * Nv, No * Nv, generator=g, **f8).mul_(sigma_eri)
    ovov = (ovov.triu() + ovov.triu(1).T).reshape(No, Nv, No, Nv).contiguous()
    ooov = torch.randn(No, No, No * Nv, generator=g, **f8).mul_(sigma_eri)
    low = torch.ones(No, No, device="cuda").tril(-1).bool()
    ooov = torch.where(low[:, :, None], ooov.transpose(0, 1), ooov).reshape(No, No, No, Nv).contiguous()
    ovvv = torch.empty(No, Nv, Nv, Nv, **f8)
    for i in range(No):
        a = torch.randn(Nv, Nv, Nv, generator=g, **f8).mul_(sigma_eri)
        ovvv[i] = a.triu() + a.triu(1).transpose(1, 2)
    # C = s G + the pair (highest occupied, lowest virtual), s such that the dominant singular value
    # carries 90 % of the weight
    G = torch.randn(No, Nv, generator=g, **f8).cpu().numpy()
    dn = d.cpu().numpy()
    E = np.zeros((No, Nv))
    E[int(np.argmax(dn[:No])), int(np.argmin(dn[No:]))] = 1.0
    lo, hi = 0.0, 1.0
    for _ in range(45 if No > 1 else 0):
        s = 0.5 * (lo + hi)
        w = np.linalg.eigvalsh((s * G + E) @ (s * G + E).T)
        lo, hi = (s, hi) if w[-1] > 0.9 * w.sum() else (lo, s)
    C = 0.5 * (lo + hi) * G + E
    C = torch.from_numpy(C / (math.sqrt(2.0) * np.linalg.norm(C))).cuda()
    return {"F": F, "ovov": ovov, "ooov": ooov, "ovvv": ovvv, "C": C}


def _mask(No, Nv):
    """The slots of the five blocks that are amplitudes."""
    m = torch.ones(5, No, No, Nv, Nv, dtype=torch.bool, device="cuda")
    o, v = torch.arange(No, device="cuda"), torch.arange(Nv, device="cuda")
    for k in (0, 2, 3):
        m[k, o, o] = False
        m[k][:, :, v, v] = False
    m[2, 0] = m[2, :, 0] = False
    m[2, :, :, 0] = m[2, :, :, :, 0] = False
    m[4, :, 0] = m[4, :, :, :, 0] = False
    m[4, 0, :, 0] = False
    return m


def _vector(No, Nv, seed):
    """A vector of the first-order space with the symmetries of the singlet, amplitudes N(0, 1e-2)."""
    x = torch.randn(5, No, No, Nv, Nv, generator=_gen(seed, 77), dtype=torch.float64, device="cuda").mul_(1e-2)
    for k in (0, 2, 3):
        t = x[k] - x[k].transpose(0, 1)
        x[k] = 0.5 * (t - t.transpose(2, 3))
    x[1] = 0.5 * (x[1] + x[1].transpose(0, 1).transpose(2, 3))
    return x.mul_(_mask(No, Nv)).contiguous()


def _contraction_inputs(case, seed):
    S, Nv = case["S"], case["Nv"]
    g, f8 = _gen(seed, 5), dict(dtype=torch.float64, device="cuda")
    x = torch.randn(S, Nv, Nv, generator=g, **f8).mul_(1e-2)
    Fv = torch.randn(Nv, Nv, generator=g, **f8).mul_(1e-3)
    Fv = Fv + Fv.T
    Fv.diagonal().copy_(torch.rand(Nv, generator=g, **f8) * 2.8 + 0.2)
    return x, Fv.contiguous()


def _handle(inst, shift=0.0):
    return esmp2.Handle(inst["F"], inst["ovov"], inst["ooov"], inst["ovvv"], inst["C"], level_shift=shift)


def prepare(case, seed):
    k = case["kind"]
    if k == "contraction":
        x, Fv = _contraction_inputs(case, seed)
        return {"case": case, "x": x, "F": Fv, "y": torch.empty_like(x)}
    if k == "batch":
        insts = [_instance(No, Nv, seed + 7919 * n) for n, (No, Nv) in enumerate(_shapes(case))]
        return {"case": case, "instances": [{n: t.cpu().numpy() for n, t in i.items()} for i in insts]}
    inst = _instance(case["No"], case["Nv"], seed, case.get("sigma_off", 1e-3))
    if k == "sigma":   # the program keeps the handle, its vector and the output
        h = _handle(inst)
        return {"case": case, "h": h, "x": _vector(case["No"], case["Nv"], seed), "y": h.empty()}
    if k == "gradient":   # a state solved as far as float64 goes
        h = _handle(inst)
        h.solve(tol=1e-12, maxit=2000, precision=esmp2.MIXED_BF16)
        return {"case": case, "h": h}
    return {"case": case, "inst": inst}


# ------------------------------------------------------------------------------------ one pass
def run(state):
    case = state["case"]
    k = case["kind"]
    if k == "contraction":
        st = esmp2.virtual_contraction_noalloc(state["x"], state["F"], state["y"], case["S"], case["Nv"],
                                               torch.cuda.current_stream())
        if st != esmp2.OK:
            raise RuntimeError("virtual_contraction_noalloc: status %d" % st)
        return state["y"]
    if k == "sigma":
        return state["h"].sigma(state["x"], PRECISION[case["precision"]], out=state["y"])
    if k == "solve":
        h = _handle(state["inst"], case["shift"])
        try:
            h.solve(tol=case["tol"], maxit=2000, precision=PRECISION[case["precision"]])
            out = {"energy": h.energy()}
            if case["solution"]:
                out["x"] = h.solution()
        finally:
            h.close()
        return out
    if k == "batch":
        st, res = esmp2.batch_solve(state["instances"], tol=case["tol"], precision=PRECISION[case["precision"]],
                                    concurrency=case["concurrency"])
        if st != esmp2.OK:
            raise RuntimeError("batch_solve: status %d" % st)
        return [{n: r[n] for n in ("E2", "E2_D", "E2_L", "E2_S")} for r in res]
    if k == "gradient":
        dF, dov, _ = state["h"].grad()
        return {"dF": dF, "dOVOV": dov}
    i = state["inst"]
    F, ovov = i["F"].detach().requires_grad_(True), i["ovov"].detach().requires_grad_(True)
    e = esmp2_energy(F, ovov, i["ooov"], i["ovvv"], i["C"], case["tol"], PRECISION[case["precision"]])
    e.backward()
    return {"E2": e.detach(), "dF": F.grad, "dOVOV": ovov.grad}


# ------------------------------------------------------------------------------------ the work
def _unique(No, Nv):
    """Amplitudes that no symmetry gives: T, X, Y with i < j and a < b, the S pairs once, Z whole."""
    return 3 * (No * (No - 1) // 2) * (Nv * (Nv - 1) // 2) + No * No * Nv * Nv / 2 + No * No * Nv * Nv


def _sigma_flops(No, Nv):
    return 4.0 * _unique(No, Nv) * (No + Nv)


def _solve_work(No, Nv):
    """Input blocks read, integral transforms, and about ten operator applications."""
    N = No + Nv
    inputs = 8.0 * (N * N + (No * Nv) ** 2 + No ** 3 * Nv + No * Nv ** 3)
    transforms = 2.0 * (No * Nv ** 3 * No + No * No * Nv ** 3 * 4 + 4 * No ** 4 * Nv)
    return inputs, transforms + 10.0 * _sigma_flops(No, Nv)


def work(case):
    k = case["kind"]
    if k == "contraction":
        S, Nv = case["S"], case["Nv"]
        return {"bytes": 8.0 * (2 * S * Nv * Nv + Nv * Nv), "flops": 4.0 * S * Nv ** 3}
    if k == "batch":
        w = [_solve_work(*s) for s in _shapes(case)]
        return {"bytes": sum(b for b, _ in w), "flops": sum(f for _, f in w)}
    No, Nv = case["No"], case["Nv"]
    n = 5 * No * No * Nv * Nv
    if k == "sigma":
        return {"bytes": 16.0 * n, "flops": _sigma_flops(No, Nv)}
    back = 8.0 * (n + 2 * (No * Nv) ** 2 + 2 * (No + Nv) ** 2)   # read x, write dF and dOVOV
    if k == "gradient":
        return {"bytes": back, "flops": _sigma_flops(No, Nv)}
    b, f = _solve_work(No, Nv)
    if k == "training":
        return {"bytes": b + back, "flops": f + _sigma_flops(No, Nv)}
    return {"bytes": b + (8.0 * n if case["solution"] else 0.0), "flops": f}


# ------------------------------------------------------------------------------------ in 64 bits
# The same quantities from the textbook formulas, in plain float64 torch.
def _top(F, C):
    """Occupied and virtual rotations of the transition-orbital-pair basis and the singular values."""
    No, Nv = C.shape
    C = C / (math.sqrt(2.0) * C.norm())
    _, s, Vh = torch.linalg.svd(C, full_matrices=False)
    V = Vh.T.contiguous()
    V = V * torch.sign(V.gather(0, V.abs().argmax(0, keepdim=True)))
    U = (C @ V) / s
    A, Q = V.clone(), torch.eye(Nv, dtype=torch.float64, device=F.device)
    for k in range(No):   # Householder reflectors that triangularise V complete the virtual space
        w = torch.zeros(Nv, dtype=torch.float64, device=F.device)
        w[k:] = A[k:, k]
        w[k] += (1.0 if A[k, k] >= 0 else -1.0) * A[k:, k].norm()
        w = w / w.norm()
        A = A - 2.0 * torch.outer(w, w @ A)
        Q = Q - 2.0 * torch.outer(Q @ w, w)
    return U, torch.cat([V, Q[:, No:]], 1), s


class _Reference:
    """The first-order equation of one state; F and ovov may require gradients."""

    def __init__(self, inst, shift, F=None, ovov=None):
        F = inst["F"] if F is None else F
        ovov = inst["ovov"] if ovov is None else ovov
        self.No, self.Nv = inst["C"].shape
        No, Nv = self.No, self.Nv
        U, W, self.lam = _top(inst["F"], inst["C"])
        R = torch.block_diag(U, W)
        self.F = R.T @ F @ R
        self.g = torch.einsum("iajb,ip->pajb", ovov, U)
        self.g = torch.einsum("pajb,aq->pqjb", self.g, W)
        self.g = torch.einsum("pqjb,jr->pqrb", self.g, U)
        self.g = torch.einsum("pqrb,bs->pqrs", self.g, W)
        ooov = torch.einsum("ijka,ip,jq,kr,as->pqrs", inst["ooov"], U, U, U, W)
        ovvt = torch.matmul(inst["ovvv"], W[:, :No].contiguous())                 # (ia|bu')
        ovvt = torch.einsum("iabu,ip->pabu", ovvt, U)
        self.ovvt = torch.einsum("pabu,aq,br->pqru", ovvt, W, W)
        self.ooov = ooov
        lam, Fd = self.lam, self.F.diagonal()
        self.omega = (2.0 * lam ** 2 * (Fd[No:2 * No] - Fd[:No])).sum() - shift
        self.mask = _mask(No, Nv).to(torch.float64)

    def rhs(self):
        No, Nv, lam, g, F = self.No, self.Nv, self.lam, self.g, self.F
        oo, vt = self.ooov, self.ovvt
        w = 2.0 * lam ** 2
        u = torch.arange(No, device=lam.device)
        f0 = F[:No, No:].T                                                        # [a][j]
        f0 = f0 + torch.einsum("u,uja->aj", w, oo[u, u]) - 0.5 * torch.einsum("u,uja->aj", w, oo[u, :, u])
        f0 = f0 - torch.einsum("u,jau->aj", w, vt[:, :, u, u]) + 0.5 * torch.einsum("u,uja->aj", w, vt[:, u, :, u])
        D = torch.zeros(No, Nv, dtype=lam.dtype, device=lam.device)               # singles of Psi0
        D[u, u] = lam
        e = torch.einsum
        dT = e("ia,bj->ijab", D, f0)
        Q = vt.permute(0, 3, 2, 1)                                                # Q[j][i][a][b] = (jb|ai')
        lq = lam[:, None, None, None] * Q.transpose(0, 1)                         # lam_i Q_ji[a][b]
        oa = torch.zeros(No, No, Nv, Nv, dtype=lam.dtype, device=lam.device)
        oa[:, :, :No] = e("a,aijb->ijab", lam, oo)                                # lam_a (ai|jb)
        anti = lambda t: t - t.transpose(2, 3)  # noqa: E731
        swap = lambda t: t.transpose(0, 1)  # noqa: E731
        T = anti(dT - swap(dT)) + anti(lq - swap(lq)) - anti(oa - swap(oa))
        S = dT + swap(dT).transpose(2, 3) + lq + swap(lq).transpose(2, 3) - oa - swap(oa).transpose(2, 3)
        gv = g.permute(0, 2, 1, 3)                                                # [i][j][a][b] = (ia|jb)

        def pair(q):
            t = e("ia,jb->ijab", D, q)
            return anti(t - swap(t))
        XY = lam[0] * (gv - swap(gv))
        X = XY + pair(g[0, 0] - g[:, 0, 0, :])
        Y = XY + pair(g[0, 0])
        Z = lam[0] * gv + e("jb,ia->ijab", D, g[:, :, 0, 0]) + e("ia,jb->ijab", D, g[:, :, 0, 0] - g[0, :, :, 0].T)
        return torch.stack([T, S, X, Y, Z]) * self.mask

    def sigma(self, x):
        No, F = self.No, self.F
        e = torch.einsum
        Fo, Fv, f = F[:No, :No], F[No:, No:], F[:No, No:]
        T, S, X, Y, Z = x
        y = torch.matmul(x, Fv) + torch.matmul(Fv, x)
        y = y - e("li,kljab->kijab", Fo, x) - e("lj,kilab->kijab", Fo, x) - self.omega * x
        f00, pair = f[0, 0], Fv[0, 0] - Fo[0, 0]
        VX, WZ = e("c,ijcb->ijb", f[0], X), e("c,ijac->ija", f[0], Z)
        G, H = e("kc,kjcb->jb", f, X + Z), e("kc,ikac->ia", f, Y + Z)
        OX, OZ = e("k,kjab->jab", f[:, 0], X), e("k,qkab->qab", f[:, 0], Z)
        CYZ = e("d,kdc->kc", Fv[0], Z[0]) - e("l,lkc->kc", Fo[:, 0], Z[:, :, 0])
        anti = lambda t: t - t.transpose(2, 3)  # noqa: E731
        swap = lambda t: t.transpose(0, 1)  # noqa: E731
        zero = torch.zeros_like(T)

        def put(t, *at):
            r = zero.clone()
            r[at] = t
            return r
        a = slice(None)
        yT = f00 * (X + Y) - anti(put(VX, a, a, 0)) - put(OX, 0) + put(OX, a, 0)
        gT = put(G, 0, a, 0)
        yT = yT + anti(gT - swap(gT))
        hS, wS = put(H, 0, a, 0), put(WZ, a, a, a, 0)
        oS = put(OZ, a, 0)
        yS = f00 * (Z + swap(Z).transpose(2, 3))
        for t in (hS - swap(wS).transpose(2, 3), -oS):
            yS = yS + t + swap(t).transpose(2, 3)
        T0, S0 = T[0], S[0]
        yX = f00 * T - anti(e("a,ijb->ijab", f[0], T[:, :, 0])) + pair * X
        tX = -e("i,jab->ijab", f[:, 0], T0) + anti(e("ia,jb->ijab", f, T0[:, 0]))
        yX = yX + tX - swap(tX)
        tY = anti(e("ia,jb->ijab", f, S0[:, 0])) + anti(put(CYZ, 0, a, 0))
        yY = f00 * T + tY - swap(tY) + pair * Y
        yZ = f00 * S - e("b,ija->ijab", f[0], S[:, :, :, 0]) - e("j,iab->ijab", f[:, 0], S[:, 0])
        yZ = yZ + e("jb,ia->ijab", f, S[:, 0, :, 0]) + e("ia,jb->ijab", f, T0[:, 0]) + pair * Z
        yZ = yZ + put(e("a,jb->jab", Fv[:, 0], Y[0][:, 0]), 0) - put(e("i,jb->ijb", Fo[0], Y[0][:, 0]), a, a, 0)
        return (y + torch.stack([yT, yS, yX, yY, yZ])) * self.mask

    def dot(self, u, v):
        return sum(w * (u[k] * v[k]).sum() for k, w in enumerate(WEIGHTS))

    def solve(self, b, tol=1e-13):
        """Conjugate gradients with the diagonal preconditioner."""
        No = self.No
        d = self.F.diagonal()
        D = (d[No:, None] + d[None, No:])[None, None, None] - (d[:No, None] + d[None, :No])[None, :, :, None, None] - self.omega
        D = D.expand(5, -1, -1, -1, -1).clone()
        D[2:] += self.F[No, No] - self.F[0, 0]
        x, r = torch.zeros_like(b), -b
        z = r / D
        p, rz, bb = z.clone(), self.dot(r, z), float(self.dot(b, b))
        for _ in range(400):
            q = self.sigma(p)
            al = rz / self.dot(p, q)
            x, r = x + al * p, r - al * q
            if float(self.dot(r, r)) <= tol * tol * bb:
                break
            z = r / D
            new = self.dot(r, z)
            p, rz = z + (new / rz) * p, new
        return x

    def parts(self, b, x):
        q = self.sigma(x)
        return [w * (2.0 * (b[k] * x[k]).sum() + (x[k] * q[k]).sum()) for k, w in enumerate(WEIGHTS)]

    def small_triples(self, chunk):
        """E2_S in pieces: -2 sum b_I^2 / D_I over the triples without the pair t -> t', hole by hole."""
        No, Nv, lam, g = self.No, self.Nv, self.lam, self.g
        d = self.F.diagonal()
        v = d[No:]
        vvv = v[:, None, None] + v[None, :, None] + v[None, None, :]
        gv = g.permute(0, 2, 1, 3)

        def drop(t, axes):
            for ax in axes:
                t.select(ax, 0).zero_()

        def same(i, j, k):
            b = torch.zeros(Nv, Nv, Nv, dtype=v.dtype, device=v.device)
            for s, p, q, h in ((1, i, j, k), (-1, k, j, i), (-1, i, k, j)):
                V = s * lam[h] * (gv[p, q] - gv[q, p])
                b[:, :, h] += V
                b[h] -= V.T
                b[:, h] -= V
            if 0 in (i, j, k):
                drop(b, (0, 1, 2))
            return -(b * b / (vvv - d[i] - d[j] - d[k] - self.omega)).sum() / 3.0

        def mixed(i, j, k):
            b = torch.zeros(Nv, Nv, Nv, dtype=v.dtype, device=v.device)
            b[:, :, k] += lam[k] * gv[i, j]
            b[:, k] -= lam[k] * gv[i, j]
            b[:, :, j] -= lam[j] * gv[i, k]
            b[:, j] += lam[j] * gv[i, k]
            b[i] += lam[i] * (gv[k, j] - gv[j, k]).T
            if i == 0:
                drop(b, (0,))
            if j == 0:
                drop(b, (1, 2))
            return -(b * b / (vvv - d[i] - d[j] - d[k] - self.omega)).sum()

        jobs = [(same, i, j, k) for i in range(No) for j in range(i + 1, No) for k in range(j + 1, No)]
        jobs += [(mixed, i, j, k) for i in range(No) for j in range(No) for k in range(j + 1, No)]
        for n in range(0, len(jobs), chunk):
            yield sum(fn(i, j, k) for fn, i, j, k in jobs[n:n + chunk])


def _energies(inst, shift, with_x):
    ref = _Reference(inst, shift)
    b = ref.rhs()
    x = ref.solve(b)
    e = [float(t) for t in ref.parts(b, x)]
    es = float(sum(ref.small_triples(64))) if ref.No > 1 else 0.0
    out = {"E2_D": e[0] + e[1], "E2_L": e[2] + e[3] + e[4], "E2_S": es}
    out["E2"] = out["E2_D"] + out["E2_L"] + es
    return (out, x) if with_x else out


def _gradient(inst):
    with torch.no_grad():
        ref = _Reference(inst, 0.0)
        x = ref.solve(ref.rhs())
        e2 = sum(float(t) for t in ref.parts(ref.rhs(), x)) + float(sum(ref.small_triples(64)))
    F, ovov = inst["F"].clone().requires_grad_(True), inst["ovov"].clone().requires_grad_(True)
    ref = _Reference(inst, 0.0, 0.5 * (F + F.T), 0.5 * (ovov + ovov.permute(2, 3, 0, 1)))
    top = [ref.F, ref.g]   # the functional is stationary in x: x stays fixed
    acc = torch.autograd.grad(sum(ref.parts(ref.rhs(), x)), top, retain_graph=True, allow_unused=True)
    acc = [torch.zeros_like(t) if a is None else a for a, t in zip(acc, top)]
    for e in ref.small_triples(8):
        for a, t in zip(acc, torch.autograd.grad(e, top, retain_graph=True, allow_unused=True)):
            if t is not None:
                a += t
    dF, dov = torch.autograd.grad(top, [F, ovov], acc)
    return e2, dF, dov


def exact(case, seed):
    k = case["kind"]
    if k == "contraction":
        x, Fv = _contraction_inputs(case, seed)
        return torch.matmul(x, Fv) + torch.matmul(Fv, x)
    if k == "batch":
        return [_energies(_instance(No, Nv, seed + 7919 * n), 0.0, False) for n, (No, Nv) in enumerate(_shapes(case))]
    No, Nv = case["No"], case["Nv"]
    if No * No * Nv * Nv > 5e7 or No * (Nv ** 3) > 2.5e8:   # over about 20 seconds
        return None
    inst = _instance(No, Nv, seed, case.get("sigma_off", 1e-3))
    if k == "sigma":
        return _Reference(inst, 0.0).sigma(_vector(No, Nv, seed))
    if k == "solve":
        e, x = _energies(inst, case["shift"], True)
        return {"energy": e, "x": x} if case["solution"] else {"energy": e}
    e2, dF, dov = _gradient(inst)
    return {"dF": dF, "dOVOV": dov} if k == "gradient" else {"E2": e2, "dF": dF, "dOVOV": dov}
