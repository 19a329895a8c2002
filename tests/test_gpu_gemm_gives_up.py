"""A GEMM whose waits run out: a build of its own in which every wait inside the pipelines gives up at its first poll. The
kernels must report it, end their copies and tensor-core instructions in flight, and leave the GPU usable."""
import ctypes
import os
import subprocess

import pytest
import torch

pytestmark = pytest.mark.gpu

STUB = r"""
#include "ssa_host.h"
namespace ssa {
ssa_status set_error(ssa_status code, const char *) { return code; }
}
"""


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    from paper_2602_19775_gb300 import build
    d = tmp_path_factory.mktemp("gemm")
    (d / "stub.cu").write_text(STUB)
    out = str(d / "libgemm.so")
    subprocess.check_call([build._nvcc(), *build.ARCH, *build.NVCC_FLAGS, "-DSSA_TC_WAIT_LIMIT=0", "-I", build.CSRC, "-shared",
                           "-o", out, os.path.join(build.CSRC, "ssa_tc_gemm.cu"), str(d / "stub.cu"), "-lcudart"])
    return ctypes.CDLL(out)


# one K block, fewer blocks than stages, many tiles, and K split over the SMs
@pytest.mark.parametrize("M,N,K,split", [(128, 128, 64, False), (300, 500, 192, False), (2304, 4000, 1024, False),
                                         (256, 512, 4096, True)])
def test_gemm_gives_up(lib, M, N, K, split):
    from paper_2602_19775_gb300 import ssa
    a = torch.randn((M, K), device="cuda").to(torch.bfloat16)
    b = torch.randn((N, K), device="cuda").to(torch.bfloat16)
    d = torch.zeros((M, N), device="cuda")
    err = torch.zeros(1, dtype=torch.int32, device="cuda")
    p = lambda t: ctypes.c_void_p(t.data_ptr())
    lib.ssa_bf16_gemm_work_words.restype = ctypes.c_int64
    words = int(lib.ssa_bf16_gemm_work_words(M, N, K)) if split else 0
    assert (words > 0) == split
    work = torch.zeros(max(words, 1), dtype=torch.float64, device="cuda")
    assert lib.ssa_bf16_gemm(p(a), p(b), M, N, K, K, K, None, p(d), N, p(work) if split else None,
                             ctypes.c_int64(words), p(err), ctypes.c_void_p(torch.cuda.current_stream().cuda_stream)) == 0
    torch.cuda.synchronize()
    assert err.item() != 0
    # the library's own call, with the ordinary limit, right after it
    ref = a.double() @ b.double().T
    assert (ssa.bf16_gemm(a, b).double() - ref).abs().max() <= K * 2.0 ** -24 * (a.double().abs() @ b.double().abs().T).max()
