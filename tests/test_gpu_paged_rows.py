"""Paged head: rows of a tile go to their slots from the staged tile.  Every row at a slot of
its own (no runs), rows at the edges of the 128-row boxes, both head widths (runs of 32 and
of 16 columns), with and without R_M: bit for bit the in-place head's rows, and nothing else
written."""
import numpy as np
import pytest
import torch

from paper_2609_35139_gb300 import RepairSession, cr
from paper_2609_35139_gb300.session import Assembled

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("rope", [False, True])
@pytest.mark.parametrize("dh, heads", [(64, 4), (128, 2), (64, 8)])
@pytest.mark.parametrize("n", [1, 31, 127, 128, 129, 256, 389])
def test_scattered_rows(n, dh, heads, rope):
    layers, d_b = 2, 256
    t = cr.target_dims(layers, heads, dh, 128, "bf16")
    r = cr.repairer_dims(8, 64, d_b, 0, 4, 256, 1e-5, 1e4)
    d_kv, plane = 2 * layers * heads * dh, heads * dh
    g = torch.Generator("cuda").manual_seed(n + dh)
    rand = lambda *s: torch.randn(s, generator=g, device="cuda")  # noqa: E731
    w = {"w_out": (rand(d_kv, d_b) / 16).to(torch.bfloat16), "b_out": rand(d_kv),
         "sigma_stale": rand(d_kv).abs() + 0.5, "sigma_delta": rand(d_kv).abs() + 0.5}
    sess = RepairSession(t, r, cr.PackedWeights(w, 0), n)
    stale = rand(n, d_kv).to(torch.bfloat16)
    sess.kv.copy_(stale)
    sess.yf.copy_(rand(n, d_b).to(torch.bfloat16))
    sess.pos.copy_(torch.arange(n, dtype=torch.int32, device="cuda") * 7)
    num_slots = 2 * n + 5
    slots = np.random.default_rng(n).permutation(num_slots)[:n].astype(np.int64)
    slots[::5] = -1
    inv = (1e4 ** (-2.0 * np.arange(dh // 2) / dh)).astype(np.float32) if rope else None
    mode = cr.CR_ROPE_GLOBAL if rope else cr.CR_ROPE_NONE
    paged = torch.full((2 * layers, num_slots, plane), 0x7F7F, dtype=torch.int16, device="cuda")
    sess.apply_paged(Assembled(n, np.asarray([0, n], np.int32)), torch.from_numpy(slots).cuda(),
                     paged.view(torch.bfloat16), num_slots, inv, mode)
    ref = stale.clone()
    cr.cr_apply_residual(sess.target, sess.rep, sess.weights, sess.yf, n, ref, sess.pos, inv, mode,
                         workspace=sess.workspace)
    want = torch.full_like(paged, 0x7F7F)
    keep = torch.from_numpy(slots >= 0).cuda()
    at = torch.from_numpy(slots[slots >= 0]).cuda()
    want[:, at] = ref.view(torch.int16).reshape(n, 2 * layers, plane)[keep].transpose(0, 1)
    assert torch.equal(paged, want)
    assert torch.equal(sess.kv, stale)
