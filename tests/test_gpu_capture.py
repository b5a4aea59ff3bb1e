"""A float64 operator application captured in a CUDA graph stays valid: what other calls on the handle
allocate later does not move the buffers it works on."""
import pytest

import synth
from tests.gpu_util import handle_for, random_block_vector

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec", ["fp64", "fp64_tc"])
@pytest.mark.parametrize("No,Nv", [(1, 20), (5, 18), (17, 36), (33, 36)])
def test_captured_sigma_survives_other_calls(No, Nv, prec):
    import torch
    from paper_2003_12923_gb300 import esmp2
    p = {"fp64": esmp2.FP64, "fp64_tc": esmp2.FP64_TC}[prec]
    stream = torch.cuda.Stream()
    inst = synth.make_instance(No, Nv, 1)
    h = esmp2.Handle(inst["F"], inst["ovov"], inst["ooov"], inst["ovvv"], inst["C"], stream=stream)
    x = torch.from_numpy(random_block_vector(No, Nv, 7)).cuda()
    y = torch.zeros_like(x)
    torch.cuda.synchronize()
    with torch.cuda.stream(stream):
        h.sigma(x, p, out=y)
        ref = y.clone()
    torch.cuda.synchronize()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g, stream=stream):
        h.sigma(x, p, out=y)
    # calls with larger and other workspaces, and a vector's worth of memory that they may have given back
    for q in (esmp2.FP64_TC, esmp2.FP64):
        h.virtual_contraction(x, q)
    for q in (esmp2.MIXED_BF16, esmp2.FP64_TC, esmp2.FP64) + ((esmp2.REDUCED_MIXED,) if No <= 32 else ()):
        h.solve(tol=1e-8, maxit=500, precision=q)
        h.solution()
    h2 = handle_for(inst)
    h2.solve(tol=1e-8, maxit=500, precision=esmp2.MIXED_BF16)
    torch.cuda.synchronize()
    b2 = h2.rhs()
    y.zero_()
    torch.cuda.synchronize()
    g.replay()
    torch.cuda.synchronize()
    assert torch.equal(y, ref)
    e = h2.energy()["E2"]
    h3 = handle_for(inst)
    h3.solve(tol=1e-8, maxit=500, precision=esmp2.MIXED_BF16)
    assert torch.equal(h2.rhs(), b2) and h3.energy()["E2"] == e   # nothing of the other handle was written
    for k in (h, h2, h3):
        k.close()
