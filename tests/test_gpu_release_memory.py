"""Memory that closed handles leave with the library: returned on request, and before an allocation of the library's own fails."""
import ctypes

import pytest
import torch

from paper_2211_07572_gb300 import _lib, inputs
from paper_2211_07572_gb300.solver import GraphBatch, SlabSolver, release_memory

pytestmark = pytest.mark.gpu
GIB = 1 << 30


def _free():
    torch.cuda.synchronize()
    torch.cuda.empty_cache()
    return torch.cuda.mem_get_info()[0]


def _close_a_handle():
    """Factor and close a handle of about 13 GiB; returns what it held."""
    s = SlabSolver(2, 2048, 32, inputs.POISSON, precision="fp32")
    held = s.device_bytes
    s.close()
    return held


def test_release_memory_returns_what_closed_handles_held():
    release_memory()
    before = _free()
    held = _close_a_handle()
    assert _free() <= before - held // 2                     # kept for the next handle
    release_memory(2 * GIB)
    assert before - 3 * GIB <= _free() <= before - GIB       # (the driver rounds to its own pieces)
    release_memory()
    assert _free() >= before - GIB // 4
    assert _lib.load().slab_release_memory(-1) == _lib.SLAB_EINVAL


@pytest.mark.parametrize("what", ["batch", "product", "handle"])
def test_an_allocation_that_needs_the_kept_memory(what):
    """All but 3 GiB of the free memory belongs to another allocator: what closed handles left must go back first."""
    release_memory()
    held = _close_a_handle()
    ballast = None
    try:
        ballast = torch.empty(_free() - 3 * GIB, dtype=torch.uint8, device="cuda")
        assert held > 10 * GIB
        if what == "batch":
            B = GraphBatch([1024] * 2, b=16)
            assert 4 * GIB < B.device_bytes < held
            B.close()
        elif what == "handle":
            s = SlabSolver(2, 1536, 32, inputs.POISSON, precision="fp64")     # another size: other pieces
            assert s.device_bytes > 4 * GIB
            s.close()
        else:                                                # the product's scratch: 4 (M + N) K bytes
            M, N, K = 640, 640, 1 << 20
            a = torch.ones(M, K, device="cuda")              # 2.5 GiB, from what is left; B is A
            c = torch.zeros(M, N, device="cuda")
            err = torch.zeros(1, dtype=torch.int32, device="cuda")
            P = lambda t: ctypes.c_void_p(t.data_ptr())
            st = _lib.load().slab_tc_gemm(M, N, K, 1.0, P(a), K, P(a), K, 0.0, P(c), N, 0, 2, P(err), None)
            torch.cuda.synchronize()
            assert st == _lib.SLAB_OK and int(err) == 0 and bool((c == float(K)).all())
    finally:
        del ballast
        torch.cuda.empty_cache()
        release_memory()


def test_what_is_kept_follows_use():
    """One large handle, then small ones: each round with no handle left lowers the kept memory by a quarter.  (3/4)^13 of 13 GiB
    is 0.3 GiB; the driver's pieces and the small handles make up the rest of the bound."""
    release_memory()
    before = _free()
    held = _close_a_handle()
    kept = before - _free()
    assert held // 2 <= kept <= held + held // 4 + GIB // 4
    for _ in range(13):
        s = SlabSolver(2, 128, 16, inputs.POISSON, precision="fp32")
        s.close()
        torch.cuda.synchronize()
    assert before - _free() <= GIB
    release_memory()


def test_never_more_than_a_quarter_of_the_device_is_kept():
    release_memory()
    before = _free()
    s = SlabSolver(2, 4096, 32, inputs.POISSON, precision="fp32", stage2="oddeven")
    total = torch.cuda.mem_get_info()[1]
    assert s.device_bytes > total // 3
    s.close()
    assert total // 8 <= before - _free() <= total // 4 + GIB // 4
    release_memory()
