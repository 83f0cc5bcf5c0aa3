"""The fp32 residual add at each tile width and walk that its rule picks: the same bits as
the same rows in short calls."""
import pytest
import torch

from paper_2609_35139_gb300 import cr

pytestmark = pytest.mark.gpu


# (rows, columns, depth) for 128-wide, 160-wide and 256-wide tiles, and 256-wide ones in
# bands because the tile updated in place shares L2 with A; one column tile, which has no
# bands, however large A is; ragged rows and columns
@pytest.mark.parametrize("M,N,K", [(3001, 2048, 512), (5119, 2048, 520), (9001, 1008, 1024), (60001, 528, 512),
                                   (9001, 4096, 1032), (70001, 128, 512)])
def test_residual_add_widths(M, N, K):
    g = torch.Generator("cuda").manual_seed(M + N)
    A = torch.randn(M, K, generator=g, device="cuda").to(torch.bfloat16)
    W = (torch.randn(N, K, generator=g, device="cuda") / K ** 0.5).to(torch.bfloat16)
    b = torch.randn(N, generator=g, device="cuda")
    start = torch.randn(M, N, generator=g, device="cuda")
    whole, parts = start.clone(), start.clone()
    cr.cr_linear(A, W, b, whole, cr.CR_EPI_ADD_F32)
    for r in range(0, M, 768):
        cr.cr_linear(A[r:r + 768], W, b, parts[r:r + 768], cr.CR_EPI_ADD_F32)
    torch.cuda.synchronize()
    assert torch.equal(whole, parts)
    # fp32 accumulation of K bf16 products of unit variance
    want = A.double() @ W.double().T + b.double() + start.double()
    assert float((whole.double() - want).abs().max()) <= 1e-3
