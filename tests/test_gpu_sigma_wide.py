"""The residual statistic over rows of 128 KB, whose blocks are wider from 2048 tokens on: both
sides of that line and a ragged last slice, against float64."""
import pytest
import torch

from paper_2609_35139_gb300 import cr

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("L,H,n", [(32, 8, 2047), (32, 8, 2048), (32, 8, 2111), (33, 8, 2177)])
def test_residual_statistic(L, H, n):
    t, D = cr.target_dims(L, H, 128, 128, "bf16"), 2 * L * H * 128
    g = torch.Generator("cuda").manual_seed(n)
    a, b = (torch.randn(n, D, generator=g, device="cuda").to(torch.bfloat16) for _ in range(2))
    got = torch.zeros(D, dtype=torch.float64, device="cuda")
    ws = torch.empty(cr.cr_sigma_workspace_bytes(t, n), dtype=torch.uint8, device="cuda")
    cr.cr_sigma_accumulate(t, a, b, n, got, ws)
    torch.cuda.synchronize()
    want = torch.zeros_like(got)
    for r in range(0, n, 512):
        want += ((a[r:r + 512].float() - b[r:r + 512].float()).double() ** 2).sum(0)
    # slices of 64 tokens summed in fp32 (a fused multiply-add each), the slices in fp64
    assert float(((got - want).abs() / want).max()) <= 64 * 2.0 ** -24
