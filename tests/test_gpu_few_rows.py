"""bf16 products of 5 to 64 rows keep what fp32 sums on the CUDA cores give, whichever kernel the
network takes for them: errors against 64 bits no larger than the few-row CUDA-core kernel's on the
same inputs, and a SiLU whose only error beside those sums is the rounding of its output."""
import pytest
import torch

from test_gpu_fused import _ll

pytestmark = pytest.mark.gpu


def _operands(M, N, Kd):
    g = torch.Generator(device="cuda").manual_seed(M * 3 + N + Kd)
    A = torch.randn((M, Kd), generator=g, device="cuda").to(torch.bfloat16)
    W = (0.02 * torch.randn((N, Kd), generator=g, device="cuda")).to(torch.bfloat16)
    return A, W


# one and two warps of rows, ragged rows and columns, 1 to 8 ways, a part of a chunk, the longest Kd
@pytest.mark.parametrize("M,N,Kd", [(5, 1024, 4096), (16, 256, 4096), (33, 1024, 2560),
                                    (64, 1024, 1024), (64, 3072, 1024), (48, 1536, 512),
                                    (31, 1000, 1992), (64, 2048, 2048), (17, 2560, 328)])
def test_few_rows_sums(M, N, Kd):
    ll = _ll()
    A, W = _operands(M, N, Kd)
    want = A.double() @ W.double().T
    err = [((ll.test_linear(A, W, torch.float32, path=p).double() - want).norm() / want.norm()).item()
           for p in (0, 2)]
    # the norm over M N >= 4096 independent roundings moves by 1 / sqrt(2 * 4096), about 1 %
    assert err[0] <= 1.03 * err[1], err


# one or two chunks a CTA, the last of them short, up to the most tiles that four CTAs each take
@pytest.mark.parametrize("M,N,Kd", [(5, 768, 256), (16, 256, 256), (64, 1024, 256), (64, 2432, 256),
                                    (33, 960, 320), (48, 696, 296), (64, 1152, 384), (17, 1344, 448)])
def test_few_rows_sums_of_short_rows(M, N, Kd):
    test_few_rows_sums(M, N, Kd)


@pytest.mark.parametrize("M,N,Kd", [(5, 512, 512), (33, 1536, 512), (64, 2048, 1024)])
@pytest.mark.parametrize("path", [0, 6])
def test_few_rows_silu(M, N, Kd, path):
    ll = _ll()
    A, W = _operands(M, N, Kd)
    bias = torch.linspace(-9, 3, N, device="cuda")
    C = ll.test_linear(A, W, torch.bfloat16, bias=bias, act=1, path=path).double()
    want = torch.nn.functional.silu(A.double() @ W.double().T + bias)
    # half an ulp of bf16's 8 significant bits (2^-8 of a value at most; tanh.approx would be 1.3 % off
    # at -4); exp and the division, some ulps of fp32 scaled by the argument (|z| <= 16: 2^-18);
    # the product's own error, 2^-20, times a slope below 1.1
    tol = want.abs() * (2.0 ** -8 + 2.0 ** -18) + 2.0 ** -19
    assert bool(((C - want).abs() <= tol).all())
