"""Linears over an A operand too large for L2 walk their tiles in bands of row tiles: the
same bits as the same rows in calls small enough for one band."""
import pytest
import torch

from paper_2609_35139_gb300 import cr

pytestmark = pytest.mark.gpu


# rows just past the 64 MB line and ragged; a W walked row tile by row tile, and one large
# enough for 20 MB bands with a last band that is not full
@pytest.mark.parametrize("M,N,K", [(16001, 512, 2048), (7900, 1168, 4104), (4100, 1536, 8192)])
@pytest.mark.parametrize("epi", [cr.CR_EPI_BF16, cr.CR_EPI_GELU_BF16, cr.CR_EPI_ADD_F32, cr.CR_EPI_F32])
def test_bands_equal_one_band(epi, M, N, K):
    g = torch.Generator("cuda").manual_seed(M + N)
    A = torch.randn(M, K, generator=g, device="cuda").to(torch.bfloat16)
    W = (torch.randn(N, K, generator=g, device="cuda") / K ** 0.5).to(torch.bfloat16)
    b = torch.randn(N, generator=g, device="cuda")
    f32 = epi in (cr.CR_EPI_ADD_F32, cr.CR_EPI_F32)
    start = torch.randn(M, N, generator=g, device="cuda")
    whole = start.clone() if f32 else torch.empty(M, N, dtype=torch.bfloat16, device="cuda")
    parts = whole.clone()
    cr.cr_linear(A, W, b, whole, epi)
    rows = int(48e6 / (2 * K)) // 256 * 256
    for r in range(0, M, rows):
        cr.cr_linear(A[r:r + rows], W, b, parts[r:r + rows], epi)
    torch.cuda.synchronize()
    assert torch.equal(whole, parts)
    want = A.double() @ W.double().T + b.double() + (start.double() if epi == cr.CR_EPI_ADD_F32 else 0)
    if epi == cr.CR_EPI_GELU_BF16:
        want = torch.nn.functional.gelu(want)
    # fp32 accumulation of K bf16 products of unit variance, one bf16 rounding where bf16
    tol = 1e-3 if f32 else 2.0 ** -8 * (want.abs() + 1)
    assert bool(((whole.double() - want).abs() <= tol).all())
