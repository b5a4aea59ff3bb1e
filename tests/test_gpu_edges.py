"""Kernels at the edges of their tiles and dispatch rules: remainders of the 32 x 32 float64 tiles
and of the 8-column rows, No on both sides of 16 and 32 (register tiles of the narrow-factor
products and of the symmetric passes), odd Nv (scalar loads), slices in one and several K chunks."""
import numpy as np
import pytest

import synth
from oracle import o2, top
from tests.gpu_util import handle_for, random_block_vector

pytestmark = pytest.mark.gpu

U64, U32 = 2.0 ** -53, 2.0 ** -24


def _torch(a):
    import torch
    return torch.from_numpy(np.ascontiguousarray(a)).cuda()


def _prep(inst, h):
    """Oracle input in the library's own TOP basis (its vectors for close singular values may
    differ from the oracle's by more than the arithmetic tested here)."""
    U, lam, Wv, F = h.top_basis()
    ovov, ooov, ovvt = top.transform_blocks(inst["ovov"], inst["ooov"], inst["ovvv"], U, Wv)
    return {"No": inst["No"], "Nv": inst["Nv"], "C": top.normalise_singles(inst["C"]), "U": U, "lam": lam,
            "Wv": Wv, "F": F, "ovov": ovov, "ooov": ooov, "ovvt": ovvt}


@pytest.mark.parametrize("singlet", [True, False])
@pytest.mark.parametrize("No,Nv,seed", [(2, 31, 1), (3, 33, 2), (5, 65, 3), (8, 97, 4), (16, 17, 5), (17, 40, 6), (33, 34, 7)])
def test_sigma_at_tile_edges(No, Nv, seed, singlet):
    from paper_2003_12923_gb300 import esmp2
    inst = synth.make_instance(No, Nv, seed, sigma_off=0.02)
    h = handle_for(inst)
    x = random_block_vector(No, Nv, seed + 50, singlet=singlet)
    ref = o2.O2(_prep(inst, h)).sigma(x)
    fmax = float(np.abs(h.top_basis()[3]).max())
    # an element sums at most K products of magnitude fmax max|x|; both sides round each of them,
    # and ten digit levels lose at most 2^-46 of the same sum
    K = 2 * No + 2 * Nv + 40
    bound = K * fmax * float(np.abs(x).max())
    for prec, rel in ((esmp2.FP64, 2 * K * U64), (esmp2.FP64_TC, 2 * K * U64 + 2.0 ** -46)):
        y = h.sigma(_torch(x), prec).cpu().numpy()
        assert np.abs(y - ref).max() <= rel * bound, (prec, np.abs(y - ref).max(), rel * bound)
    h.close()


@pytest.mark.parametrize("No,Nv,seed", [(15, 18, 1), (16, 19, 2), (17, 20, 3), (31, 34, 4), (32, 35, 5), (33, 36, 6)])
def test_rhs_at_occupied_tiles(No, Nv, seed):
    inst = synth.make_instance(No, Nv, seed)
    h = handle_for(inst)
    b = h.rhs().cpu().numpy()
    ref = o2.O2(_prep(inst, h)).rhs()
    # at most eight integrals each; a rotated integral sums at most No Nv gmax over its four
    # rotations, each of length <= Nv (float64 on both sides; digit products lose 2^-46 of the sum)
    gmax = max(float(np.abs(inst[k]).max()) for k in ("ovov", "ooov", "ovvv"))
    assert np.abs(b - ref).max() <= 8 * gmax * No * Nv * 4 * (2 * Nv * U64 + 2.0 ** -46)
    h.close()


@pytest.mark.parametrize("prec", ["bf16", "tf32", "reduced"])
@pytest.mark.parametrize("No,Nv,seed", [(2, 9, 1), (5, 33, 2), (7, 34, 3), (17, 37, 4)])
def test_mixed_solution_residual(No, Nv, seed, prec):
    from paper_2003_12923_gb300 import esmp2
    p = {"bf16": esmp2.MIXED_BF16, "tf32": esmp2.MIXED_TF32, "reduced": esmp2.REDUCED_MIXED}[prec]
    inst = synth.make_instance(No, Nv, seed)
    h = handle_for(inst)
    tol = 1e-9
    info = h.solve(tol=tol, maxit=2000, precision=p)
    x = h.solution()
    xn = x.cpu().numpy()
    assert info["rel_residual"] <= tol
    sym = 4 * (No + Nv) * 2.0 ** -46 * np.abs(xn).max()   # the basis change rounds each image
    for k in (0, 2, 3):
        for t in ((1, 0, 2, 3), (0, 1, 3, 2)):
            assert np.abs(xn[k] + xn[k].transpose(t)).max() <= sym
    assert np.abs(xn[1] - xn[1].transpose(1, 0, 3, 2)).max() <= sym
    # the residual by the oracle: the weights of the reported norm lie between 1/2 and 2, so the
    # unweighted ratio is at most twice the tolerance, and both sides round K products per element
    o = o2.O2(_prep(inst, h))
    b = o.rhs()
    r = b + o.sigma(xn)
    K = 2 * No + 2 * Nv + 40
    assert np.linalg.norm(r) <= 2 * tol * np.linalg.norm(b) + 2 * K * K * U64 * np.linalg.norm(xn) * np.abs(h.top_basis()[3]).max()
    h.close()


@pytest.mark.parametrize("No,Nv,seed", [(2, 9, 1), (3, 33, 2), (9, 34, 3)])
def test_gradient_of_symmetric_and_given_vectors(No, Nv, seed):
    import torch
    inst = synth.make_instance(No, Nv, seed, sigma_off=0.02)
    h = handle_for(inst)
    h.solve(tol=1e-11, maxit=2000)
    dF, dov, _ = h.grad()
    x = h.solution()
    h.set_solution(x)   # a vector of the caller's: no symmetry is assumed
    torch.cuda.synchronize()
    gF, gov, _ = h.grad()
    # the same sums in another order: a density element sums No^2 Nv products, at most 8 |x|^2 in
    # magnitude over the blocks and both images, and a rotation of both indices at most N times that
    n2 = float((x * x).sum())
    assert np.abs(np.asarray(gF) - np.asarray(dF)).max() <= (No + Nv) * No * No * Nv * U64 * 8 * n2
    # no density enters dOVOV: atomic additions in another order, then four rotations
    assert np.abs(np.asarray(gov) - np.asarray(dov)).max() <= 4 * No * Nv * U64 * np.abs(np.asarray(dov)).max()
    h.close()


@pytest.mark.parametrize("S,Nv,shift", [(1, 1, 0), (3, 7, 0), (2, 33, 0), (5, 64, 1), (1, 130, 1), (2, 257, 0)])
def test_noalloc_contraction_edges(S, Nv, shift):
    import torch
    from paper_2003_12923_gb300 import esmp2
    g = torch.Generator(device="cuda").manual_seed(S * 1000 + Nv)
    x = torch.randn(S, Nv, Nv, generator=g, device="cuda", dtype=torch.float64)
    F = torch.randn(Nv, Nv, generator=g, device="cuda", dtype=torch.float64)
    F = F + F.T
    buf = torch.full((S * Nv * Nv + 2,), 7.0, dtype=torch.float64, device="cuda")
    y = buf[shift:shift + S * Nv * Nv]   # shift 1: rows of y do not start on 16-byte boundaries
    assert esmp2.virtual_contraction_noalloc(x, F, y, S, Nv) == esmp2.OK
    xb, Fb = x.float().bfloat16().double(), F.float().bfloat16().double()
    ref = xb @ Fb + Fb @ xb
    # 2 Nv float32 additions, truncated or rounded
    bound = 2 * Nv * 2 * U32 * (xb.abs() @ Fb.abs() + Fb.abs() @ xb.abs())
    assert bool(((y.view(S, Nv, Nv) - ref).abs() <= bound + 1e-30).all())
    assert float(buf[shift + S * Nv * Nv]) == 7.0 and (shift == 0 or float(buf[0]) == 7.0)
