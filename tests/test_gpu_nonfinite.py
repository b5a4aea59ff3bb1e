"""A NaN or infinity in an integral block or in a vector never comes back as a plausible number: it
carries through the digit products of the tensor cores as NaN, to exactly the results that depend
on it.  Sizes on both sides of the narrow products' tiles (16 and 32 occupied orbitals)."""
import math

import numpy as np
import pytest

import synth
from tests.gpu_util import handle_for, random_block_vector

pytestmark = pytest.mark.gpu

SIZES = [(5, 18, 1), (17, 36, 2), (33, 36, 3)]


def _torch(a):
    import torch
    return torch.from_numpy(np.ascontiguousarray(a)).cuda()


@pytest.mark.parametrize("bad", [math.nan, math.inf])
@pytest.mark.parametrize("block,idx", [("ovov", (1, 2, 3, 4)), ("ooov", (1, 0, 2, 3)), ("ovvv", (2, 3, 4, 5))])
@pytest.mark.parametrize("No,Nv,seed", SIZES)
def test_non_finite_integral_reaches_the_result(No, Nv, seed, block, idx, bad):
    from paper_2003_12923_gb300 import esmp2
    inst = dict(synth.make_instance(No, Nv, seed))
    inst[block] = inst[block].copy()
    inst[block][idx] = bad
    h = handle_for(inst)
    assert not bool(h.rhs().isfinite().all())
    for prec in (esmp2.FP64, esmp2.MIXED_BF16) + ((esmp2.REDUCED_MIXED,) if No <= 32 else ()):
        r = h.solve(tol=1e-8, maxit=20, precision=prec, raise_on_error=False)
        assert r["status"] == esmp2.ERR_INDEFINITE or not math.isfinite(h.energy()["E2"]), (prec, r)
    h.close()


@pytest.mark.parametrize("No,Nv,seed", SIZES)
def test_non_finite_right_hand_side_is_not_converged(No, Nv, seed):
    from paper_2003_12923_gb300 import esmp2
    inst = dict(synth.make_instance(No, Nv, seed))
    inst["ooov"] = inst["ooov"].copy()
    inst["ooov"][1, 0, 2, 3] = math.nan
    h = handle_for(inst)
    precs = [esmp2.FP64, esmp2.MIXED_BF16]
    if No <= 32:
        precs += [esmp2.MIXED_TF32, esmp2.REDUCED_MIXED, esmp2.REDUCED_MINRES]
    for prec in precs:
        r = h.solve(tol=1e-8, maxit=20, precision=prec, raise_on_error=False)
        assert r["status"] in (esmp2.ERR_INDEFINITE, esmp2.ERR_NOT_CONVERGED), (prec, r)
        assert r["iterations"] <= 20 and not r["rel_residual"] <= 1e-8, (prec, r)
    h.close()


@pytest.mark.parametrize("bad", [math.nan, -math.inf])
@pytest.mark.parametrize("No,Nv,seed", SIZES)
def test_non_finite_vector_reaches_sigma(No, Nv, seed, bad):
    from paper_2003_12923_gb300 import esmp2
    h = handle_for(synth.make_instance(No, Nv, seed))
    x = random_block_vector(No, Nv, seed + 50)
    x[1, 2, 1, 3, 4] = x[1, 1, 2, 4, 3] = bad   # both images of one S amplitude
    precs = [esmp2.FP64, esmp2.FP64_TC, esmp2.MIXED_BF16]
    if No <= 32:
        precs += [esmp2.MIXED_TF32, esmp2.REDUCED_MIXED]
    for prec in precs:
        assert not bool(h.sigma(_torch(x), prec).isfinite().all()), prec
    h.close()


@pytest.mark.parametrize("bad", [math.nan, math.inf])
@pytest.mark.parametrize("No,Nv,seed", [(3, 18, 1), (2, 131, 2), (2, 200, 3)])
def test_non_finite_element_stays_in_its_row_and_column(No, Nv, seed, bad):
    from paper_2003_12923_gb300 import esmp2
    h = handle_for(synth.make_instance(No, Nv, seed))
    x = random_block_vector(No, Nv, seed + 50)
    k, i, j, a, c = 1, 1, 0, Nv - 2, Nv // 2
    # without the element the scale of the slice is the same: it is not the largest one
    x[k, i, j, a, c] = 0.0
    ref = h.virtual_contraction(_torch(x), esmp2.FP64_TC).cpu().numpy()
    x[k, i, j, a, c] = bad
    y = h.virtual_contraction(_torch(x), esmp2.FP64_TC).cpu().numpy()
    hit = np.zeros_like(y, dtype=bool)
    hit[k, i, j, a, :] = hit[k, i, j, :, c] = True
    assert np.array_equal(np.isnan(y), hit)
    assert np.array_equal(y[~hit], ref[~hit])
    h.close()
