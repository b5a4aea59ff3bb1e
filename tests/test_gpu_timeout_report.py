"""A bounded device wait that ran out reaches the caller as ESMP2_ERR_TIMEOUT through every call whose
result depends on the kernel, and the call after it succeeds.  The flag is raised by the self-test, no
wait runs out."""
import pytest

import synth
from tests.gpu_util import handle_for

pytestmark = pytest.mark.gpu


def _times_out(esmp2, call):
    with pytest.raises(esmp2.Esmp2Error) as e:
        call()
    assert e.value.args and "timed out" in str(e.value), str(e.value)


@pytest.mark.parametrize("No,Nv", [(5, 18), (17, 36), (33, 36)])
@pytest.mark.parametrize("prec", ["bf16", "tf32", "reduced", "minres", "fp64_tc"])
def test_solve_reports_a_wait_that_ran_out(No, Nv, prec):
    from paper_2003_12923_gb300 import esmp2
    if No > 32 and prec in ("tf32", "reduced", "minres"):
        pytest.skip("these forms need No <= 32")
    p = {"bf16": esmp2.MIXED_BF16, "tf32": esmp2.MIXED_TF32, "reduced": esmp2.REDUCED_MIXED,
         "minres": esmp2.REDUCED_MINRES, "fp64_tc": esmp2.FP64_TC}[prec]
    h = handle_for(synth.make_instance(No, Nv, 1))
    h.selftest_raise_timeout()
    _times_out(esmp2, lambda: h.solve(tol=1e-9, maxit=500, precision=p))
    assert h.solve(tol=1e-9, maxit=500, precision=p)["rel_residual"] <= 1e-9
    h.close()


@pytest.mark.parametrize("No,Nv", [(5, 18), (33, 36)])
def test_the_residual_that_ends_a_solve_is_checked(No, Nv):
    from paper_2003_12923_gb300 import esmp2
    h = handle_for(synth.make_instance(No, Nv, 1))
    for p in (esmp2.MIXED_BF16, esmp2.FP64_TC):
        h.solve(tol=1e-9, maxit=500, precision=p)
        h.selftest_raise_timeout()
        # the warm start is converged: its first residual ends the solve
        _times_out(esmp2, lambda: h.solve(tol=1e-8, maxit=500, precision=p))
        assert h.solve(tol=1e-8, maxit=500, precision=p)["rel_residual"] <= 1e-8
    h.close()


@pytest.mark.parametrize("No,Nv", [(5, 18), (17, 36), (33, 36)])
def test_solution_and_energy_report_a_wait_that_ran_out(No, Nv):
    import torch
    from paper_2003_12923_gb300 import esmp2
    h = handle_for(synth.make_instance(No, Nv, 1))
    for p in (esmp2.MIXED_BF16,) + ((esmp2.REDUCED_MIXED,) if No <= 32 else ()):
        h.solve(tol=1e-9, maxit=500, precision=p)
        x = h.solution()
        h.selftest_raise_timeout()
        _times_out(esmp2, h.solution)
        assert torch.equal(h.solution(), x)
    h.set_solution(x)
    h.selftest_raise_timeout()
    _times_out(esmp2, h.energy)
    assert h.energy()["E2"] < 0
    h.solve(tol=1e-9, maxit=500, precision=esmp2.MIXED_BF16)
    h.selftest_raise_timeout()
    _times_out(esmp2, h.grad)   # rotates the solution to the TOP basis
    h.close()
