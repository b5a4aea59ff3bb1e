"""The product of (ia|bc) with the transition virtuals keeps every row's own float64 accuracy, and is the
same sum when a long index is cut into ranges."""
import numpy as np
import pytest

import synth
from oracle import o2, top
from tests.gpu_util import handle_for

pytestmark = pytest.mark.gpu

U64 = 2.0 ** -53


@pytest.mark.parametrize("No,Nv,seed", [(3, 33, 1), (5, 18, 2), (16, 40, 3), (17, 36, 4)])
def test_small_rows_beside_large_ones(No, Nv, seed):
    inst = dict(synth.make_instance(No, Nv, seed))
    inst["ovov"], inst["ooov"] = np.zeros_like(inst["ovov"]), np.zeros_like(inst["ooov"])
    # rows 2^-30 of the largest one of their slice, which holds one large element at (b, c) = (Nv-1, Nv-1)
    v = inst["ovvv"] * 2.0 ** -30
    v[:, :, Nv - 1, Nv - 1] = 1.0
    inst["ovvv"] = v
    C = np.zeros((No, Nv))
    C[np.arange(No), np.arange(No)] = 0.8 ** np.arange(No)
    inst["C"] = C
    h = handle_for(inst)
    U, lam, Wv, F = h.top_basis()
    assert np.array_equal(U, np.eye(No)) and np.array_equal(Wv, np.eye(Nv))   # the rotations are exact
    b = h.rhs().cpu().numpy()
    ovov, ooov, ovvt = top.transform_blocks(inst["ovov"], inst["ooov"], inst["ovvv"], U, Wv)
    ref = o2.O2({"No": No, "Nv": Nv, "C": top.normalise_singles(C), "U": U, "lam": lam, "Wv": Wv, "F": F, "ovov": ovov,
                 "ooov": ooov, "ovvt": ovvt}).rhs()
    # S_ij^ab = lam_i (jb|ai') + lam_j (ia|bj') away from the pairs' own virtuals.  A row's product is exact
    # to 2^-53 of its largest element after each of the truncation, the join of the levels and the
    # rounding; the two rotations of the virtual indices that follow lose 2^-53 each of the largest
    # element of the block of one (i, u'), and every occupied rotation 2^-53 of its row
    out = np.abs(v[:, :, :, :No]).max()
    row = np.abs(v).max(axis=3)                                   # [i][a][b]
    S, R = b[1][:, :, No:, No:], ref[1][:, :, No:, No:]
    rows = row[:, No:, No:]
    tol = 3 * U64 * (lam[:, None, None, None] * rows.transpose(0, 2, 1)[None] + lam[None, :, None, None] * rows[:, None])
    tol = tol + 8 * U64 * out * (lam[:, None] + lam[None, :])[:, :, None, None]
    assert (np.abs(S - R) <= tol).all(), float((np.abs(S - R) / tol).max())
    h.close()


@pytest.mark.parametrize("Nv", [479, 481, 961])
def test_long_rows_in_ranges(Nv):
    import torch
    g, f8 = torch.Generator(device="cuda").manual_seed(Nv), dict(dtype=torch.float64, device="cuda")
    v = torch.randn(1, Nv, Nv, Nv, generator=g, **f8).mul_(1e-2)
    for a in range(Nv):
        v[0, a] = v[0, a].triu() + v[0, a].triu(1).T
    F = torch.diag(torch.cat([torch.full((1,), -1.0, **f8), torch.linspace(0.2, 3.0, Nv, **f8)]))
    C = torch.randn(1, Nv, generator=g, **f8)
    inst = {"F": F, "C": C, "ovvv": v, "ovov": torch.zeros(1, Nv, 1, Nv, **f8), "ooov": torch.zeros(1, 1, 1, Nv, **f8)}
    h = handle_for(inst)
    U, lam, Wv, _ = h.top_basis()
    W, l0 = torch.from_numpy(Wv).cuda(), float(lam[0]) * float(U[0, 0])
    b = h.rhs()[1, 0, 0, 1:, 1:]
    q = W.T @ torch.matmul(v[0], W[:, 0]) @ W                     # (ia|bt') in the rotated virtuals
    ref = l0 * (q + q.T)[1:, 1:]
    # three sums of Nv products on each side, each exact to 2 Nv 2^-53 (or the digits' 2^-46) of the sum of magnitudes
    m = W.abs().T @ torch.matmul(v[0].abs(), W[:, 0].abs()) @ W.abs()
    tol = abs(l0) * 3 * (2 * Nv * U64 + 2.0 ** -46) * (m + m.T)[1:, 1:]
    assert bool(((b - ref).abs() <= tol).all())
    h.close()
