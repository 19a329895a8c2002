"""The persistent GEMM over sizes that take other tile widths, lone CTAs and pairs, odd numbers of row blocks, several
rounds with a ragged last one, and operands that are used in place or copied (rows off 16 bytes, transposed), against a
float64 product of the same bf16 values; each output the sum of K exact products in binary32."""
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("M,N,K", [(2048, 2048, 64), (2176, 2304, 136), (2177, 4099, 72), (4224, 1900, 8), (129, 20000, 64),
                                   (128, 20000, 200), (2300, 2300, 65), (5000, 2000, 328)])
@pytest.mark.parametrize("layout", ["plain", "transposed", "odd rows"])
def test_tiles(M, N, K, layout):
    from paper_2602_19775_gb300 import ssa
    g = torch.Generator(device="cuda").manual_seed(M + N + K)
    if layout == "transposed":
        A = torch.randn((K, M), device="cuda", generator=g).to(torch.bfloat16).T
    elif layout == "odd rows":
        A = torch.randn((M, K + 3), device="cuda", generator=g).to(torch.bfloat16)[:, 1:K + 1]
    else:
        A = torch.randn((M, K), device="cuda", generator=g).to(torch.bfloat16)
    B = torch.randn((N, K), device="cuda", generator=g).to(torch.bfloat16)
    bias = torch.randn(N, device="cuda", generator=g)
    D = ssa.bf16_gemm(A, B, bias)
    ref = A.double() @ B.double().T + bias.double()
    bound = K * 2.0 ** -24 * (A.double().abs() @ B.double().abs().T) + 1e-6
    assert torch.all((D.double() - ref).abs() <= bound)
