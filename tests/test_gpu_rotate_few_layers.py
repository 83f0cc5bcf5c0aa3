"""The rotation of K in caches of few layers: many tokens, whose threads run over heads, too,
give the bits of the same rows in short calls, whose threads run over layers."""
import numpy as np
import pytest
import torch

from paper_2609_35139_gb300 import cr

pytestmark = pytest.mark.gpu


# layers and heads whose segments divide evenly among a token's threads and not; eight layers
# (one range), twelve (two) and twenty (four)
@pytest.mark.parametrize("L,H,dh,dtype", [(1, 8, 128, "bf16"), (2, 1, 64, "f32"), (4, 2, 64, "f32"), (7, 3, 128, "bf16"),
                                          (5, 5, 64, "bf16"), (3, 1, 128, "f32"), (8, 2, 64, "bf16"), (12, 3, 128, "f32"),
                                          (20, 1, 64, "bf16")])
@pytest.mark.parametrize("inverse", [False, True])
def test_long_call_equals_short_calls(L, H, dh, dtype, inverse):
    n, rows = 9001, 37
    t = cr.target_dims(L, H, dh, 256, dtype)
    g = torch.Generator("cuda").manual_seed(L * H + dh)
    start = torch.randn(n, 2 * L * H * dh, generator=g, device="cuda").to(torch.bfloat16 if dtype == "bf16" else torch.float32)
    pos = torch.randint(0, 4096, (n,), generator=g, device="cuda", dtype=torch.int32)
    inv = (1e6 ** (-np.arange(0, dh, 2) / dh)).astype(np.float32)
    call = cr.cr_canonicalize_chunks if inverse else cr.cr_rotate_k
    whole, parts = start.clone(), start.clone()
    call(t, whole, n, pos, inv)
    for r in range(0, n, rows):
        m = min(rows, n - r)
        call(t, parts[r:r + m], m, pos[r:r + m].clone(), inv)
    torch.cuda.synchronize()
    assert torch.equal(whole, parts)
    v = lambda x: x.view(n, L, 2, H, dh)
    assert torch.equal(v(whole)[:, :, 1], v(start)[:, :, 1])   # V untouched
    x, ang = v(start)[:, :, 0].double(), pos.double()[:, None] * torch.from_numpy(inv).cuda().double()
    c, s = ang.cos()[:, None, None], ang.sin()[:, None, None] * (-1 if inverse else 1)
    a, b = x[..., :dh // 2], x[..., dh // 2:]
    want = torch.cat([a * c - b * s, b * c + a * s], -1)
    size = (a.abs() + b.abs()).repeat(1, 1, 1, 2)
    # one rounding to the cache dtype, and the fp32 angle (up to 4096, 2^-24 relative) and products
    bound = want.abs() * (2.0 ** -8 if dtype == "bf16" else 2.0 ** -23) + size * (4096 * 2.0 ** -24 + 2.0 ** -22)
    assert bool(((v(whole)[:, :, 0].double() - want).abs() <= bound).all())
