"""Device memory a solve holds, from the counters of the device's memory pool."""
import ctypes

import pytest

import synth
from tests.gpu_util import handle_for

pytestmark = pytest.mark.gpu


class _Pool:
    def __init__(self):
        import torch
        torch.cuda.synchronize()
        try:
            self.rt = ctypes.CDLL("libcudart.so.%s" % torch.version.cuda.split(".")[0])
        except OSError:
            self.rt = ctypes.CDLL("/usr/local/cuda/lib64/libcudart.so")
        self.pool = ctypes.c_void_p()
        assert self.rt.cudaDeviceGetDefaultMemPool(ctypes.byref(self.pool), torch.cuda.current_device()) == 0

    def used(self):
        import torch
        torch.cuda.synchronize()
        v = ctypes.c_uint64()
        assert self.rt.cudaMemPoolGetAttribute(self.pool, 7, ctypes.byref(v)) == 0   # cudaMemPoolAttrUsedMemCurrent
        return v.value


    def leave(self, nbytes):
        """Take all but nbytes of the device's free memory (reserved, never touched)."""
        import gc
        import torch
        gc.collect()
        torch.cuda.synchronize()
        torch.cuda.empty_cache()
        self.rt.cudaMemPoolTrimTo.argtypes = [ctypes.c_void_p, ctypes.c_size_t]
        assert self.rt.cudaMemPoolTrimTo(self.pool, 0) == 0
        return torch.empty(torch.cuda.mem_get_info()[0] - int(nbytes), dtype=torch.uint8, device="cuda")


def test_reduced_solve_holds_no_product_vector():
    from paper_2003_12923_gb300 import esmp2
    No, Nv = 8, 80
    vec = 8 * 5 * No * No * Nv * Nv
    h = handle_for(synth.make_instance(No, Nv, 1))
    pool = _Pool()
    h.solve(tol=1e-8, maxit=500, precision=esmp2.REDUCED_MIXED)
    u = pool.used()
    h.sigma(h.rhs(), esmp2.FP64)
    # the float64 sigma is the first call to need the products, four blocks of a vector at least
    assert pool.used() - u >= 0.79 * vec
    h.close()


def test_float64_solve_gives_its_preconditioner_back():
    from paper_2003_12923_gb300 import esmp2
    No, Nv = 8, 80
    vec = 8 * 5 * No * No * Nv * Nv
    h = handle_for(synth.make_instance(No, Nv, 1))
    pool = _Pool()
    u = pool.used()
    h.solve(tol=1e-8, maxit=500, precision=esmp2.FP64)
    assert pool.used() - u <= 1.1 * vec   # the products stay
    h.close()


def test_float64_solve_without_room_for_its_preconditioner():
    import torch
    from paper_2003_12923_gb300 import esmp2
    No, Nv = 12, 160
    vec = 8 * 5 * No * No * Nv * Nv
    h = handle_for(synth.make_instance(No, Nv, 1))
    pool = _Pool()
    h.solve(tol=1e-8, maxit=500, precision=esmp2.FP64)
    zero = torch.zeros(h.shape, dtype=torch.float64, device="cuda")

    def solve():
        h.set_solution(zero)
        n = h.kernel_launches
        info = h.solve(tol=1e-8, maxit=500, precision=esmp2.FP64)
        return info["iterations"], h.kernel_launches - n

    it, launches = solve()
    x = h.solution()
    hog = pool.leave(0.5 * vec)
    assert solve() == (it, launches - 1)   # M^-1 formed in the kernels that read it, by the same formula
    del hog
    torch.cuda.empty_cache()
    assert torch.equal(h.solution(), x)
    h.close()


def test_digit_products_in_passes_where_the_planes_find_no_room():
    import torch
    from paper_2003_12923_gb300 import esmp2
    No, Nv = 12, 160
    vec = 8 * 5 * No * No * Nv * Nv
    inst = synth.make_instance(No, Nv, 1)
    h = handle_for(inst)
    x = h.rhs()
    ref = h.sigma(x, esmp2.FP64_TC)
    h.solve(tol=1e-8, maxit=500, precision=esmp2.REDUCED_MIXED)
    sol = h.solution()   # rotated back by products without a job list
    h.close()
    h = handle_for(inst)
    pool = _Pool()
    y = torch.empty_like(x)
    hog = pool.leave(1.6 * vec)   # the products' vector and less than a quarter of the planes
    h.sigma(x, esmp2.FP64_TC, out=y)
    torch.cuda.synchronize()
    del hog
    torch.cuda.empty_cache()
    assert torch.equal(y, ref)    # sums of integers: the same whatever the passes
    h.solve(tol=1e-8, maxit=500, precision=esmp2.REDUCED_MIXED)
    assert torch.equal(h.solution(), sol)
    h.close()
