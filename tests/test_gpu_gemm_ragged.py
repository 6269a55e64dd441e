"""GPU check of the persistent tensor-core linear layer where its last column tile is mostly past
N: chunks that store nothing must not let the next ones overwrite a staging buffer that a store
is still reading (seen as wrong values in the last rows of a tile, in some calls)."""
import pytest
import torch

from test_gpu_fused import _ll

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("M,N,Kd", [(40001, 320, 200), (40001, 264, 128), (19713, 320, 520)])
@pytest.mark.parametrize("dt", [torch.float32, torch.bfloat16])
def test_ragged_columns_many_tiles(M, N, Kd, dt):
    ll = _ll()
    g = torch.Generator(device="cuda").manual_seed(M + N + Kd)
    A = torch.randn((M, Kd), generator=g, device="cuda").to(torch.bfloat16)
    W = (0.05 * torch.randn((N, Kd), generator=g, device="cuda")).to(torch.bfloat16)
    want = A.double() @ W.double().T
    # fp32 sums of Kd bf16 products, and the rounding of a bf16 output
    tol = Kd * 2.0 ** -23 * Kd * 0.05 * 4 + (2.0 ** -8 * want.abs() if dt == torch.bfloat16 else 0)
    for _ in range(8):
        C = ll.test_linear(A, W, dt, path=3)
        assert bool(((C.double() - want).abs() <= tol).all())
