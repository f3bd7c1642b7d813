"""The integer-slice product keeps inside the work area that slab_fp64_tc_gemm_work_bytes asks for, and asks for what it uses."""
import ctypes

import numpy as np
import pytest
import torch

SLICES = 8


def _lib():
    from paper_2211_07572_gb300 import _lib as binding
    return binding.load()


@pytest.mark.parametrize("M,N,K", [(1, 1, 32), (200, 130, 64), (8960, 8960, 64)])
def test_work_bytes_are_16_bit_slices_and_exponents(M, N, K):
    need = SLICES * (M + N) * K * 2 + (M + N) * 4
    assert need <= int(_lib().slab_fp64_tc_gemm_work_bytes(M, N, K)) <= need + 256


@pytest.mark.gpu
@pytest.mark.parametrize("M,N,K", [(1, 9, 32), (129, 65, 64), (300, 77, 32)])
def test_nothing_is_written_behind_the_work_area(M, N, K):
    lib = _lib()
    nbytes = int(lib.slab_fp64_tc_gemm_work_bytes(M, N, K))
    area = torch.full((nbytes + 4096,), 0x5A, dtype=torch.uint8, device="cuda")     # the work area, then 4 KB that stay
    rng = np.random.default_rng(K + M)
    A, B = rng.standard_normal((M, K)), rng.standard_normal((N, K))
    Ad, Bd = torch.from_numpy(A).cuda(), torch.from_numpy(B).cuda()
    Cd = torch.zeros(M, N, dtype=torch.float64, device="cuda")
    err = torch.zeros(1, dtype=torch.int32, device="cuda")
    ptr = [ctypes.c_void_p(t.data_ptr()) for t in (Ad, Bd, Cd, area, err)]
    st = lib.slab_fp64_tc_gemm(M, N, K, 1.0, ptr[0], K, ptr[1], K, ptr[2], N, ptr[3], ptr[4],
                               ctypes.c_void_p(torch.cuda.current_stream().cuda_stream))
    torch.cuda.synchronize()
    assert st == 0 and int(err.item()) == 0
    assert bool((area[nbytes:] == 0x5A).all())
    scale = np.abs(A) @ np.abs(B).T
    assert (np.abs(Cd.cpu().numpy() - A @ B.T) / scale).max() <= 1e-13
