"""The steps of a Repair Block called one by one are the forward's, bit for bit, for bf16 and
fp32 caches, also where scores far outgrow those of a row's first key tile (so that the
attention's softmax reference matters)."""
import numpy as np
import pytest
import torch

from paper_2609_35139_gb300 import RepairSession, cr
from paper_2609_35139_gb300.session import Assembled

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("scale", [1.0, 5.0])
@pytest.mark.parametrize("mode", ["block_causal", "block_diagonal"])
@pytest.mark.parametrize("nh,hd", [(4, 64), (8, 32)])
@pytest.mark.parametrize("dtype", ["bf16", "f32"])
def test_steps_make_the_forward(dtype, nh, hd, mode, scale):
    db, hid, eps, theta = nh * hd, 4 * nh * hd, 1e-5, 1e4
    lens = [[300, 411], [90], [130, 7, 500]]
    cu = np.concatenate([[0], np.cumsum([sum(r) for r in lens])]).astype(np.int32)
    end = np.concatenate([np.repeat(np.cumsum(r), r) for r in lens]).astype(np.int32)
    n = int(cu[-1])
    g = torch.Generator("cuda").manual_seed(nh)
    rand = lambda *s: torch.randn(s, generator=g, device="cuda")  # noqa: E731
    w = {}
    for k, o, i in (("qkv", 3 * db, db), ("o", db, db), ("fc1", hid, db), ("fc2", db, hid)):
        m = rand(o, i) / i ** 0.5
        if k == "qkv":
            m[:2 * db] *= scale
        w[f"blk0.w_{k}"], w[f"blk0.b_{k}"] = m.to(torch.bfloat16), 0.02 * rand(o)
    for k in ("blk0.ln1", "blk0.ln2", "lnf"):
        w[f"{k}_g"], w[f"{k}_b"] = 1 + 0.05 * rand(db), 0.05 * rand(db)
    sess = RepairSession(cr.target_dims(4, 2, 64, 256, dtype), cr.repairer_dims(8, 64, db, 1, nh, hid, eps, theta),
                         cr.PackedWeights(w, 1), n)
    sess.h0.copy_(rand(n, db))
    sess.rein.copy_(rand(n, db))
    sess.pos.copy_(torch.cat([torch.arange(sum(r)) for r in lens]).to(torch.int32))
    sess.chunk_end.copy_(torch.from_numpy(end))
    sess.forward(Assembled(n, cu), mask_mode=mode)

    bf = lambda *s: torch.empty(s, dtype=torch.bfloat16, device="cuda")  # noqa: E731
    x, u, qkv, o, h, yf = torch.empty_like(sess.h0), bf(n, db), bf(n, 3 * db), bf(n, db), bf(n, hid), bf(n, db)
    start = torch.empty(n, dtype=torch.int32, device="cuda")
    cr.cr_chunk_starts(sess.chunk_end, cu, n, start)
    cr.cr_layernorm(sess.h0, w["blk0.ln1_g"], w["blk0.ln1_b"], eps, u, add=sess.rein, ld_add=db, x_out=x)
    cr.cr_qkv_rope(u, w["blk0.w_qkv"], w["blk0.b_qkv"], sess.pos, db, nh, theta, qkv)
    cr.cr_masked_attention(qkv, db, nh, mode, sess.chunk_end, start, cu, o)
    cr.cr_linear(o, w["blk0.w_o"], w["blk0.b_o"], x, cr.CR_EPI_ADD_F32)
    cr.cr_layernorm(x, w["blk0.ln2_g"], w["blk0.ln2_b"], eps, u)
    cr.cr_linear(u, w["blk0.w_fc1"], w["blk0.b_fc1"], h, cr.CR_EPI_GELU_BF16)
    cr.cr_linear(h, w["blk0.w_fc2"], w["blk0.b_fc2"], x, cr.CR_EPI_ADD_F32)
    cr.cr_layernorm(x, w["lnf_g"], w["lnf_b"], eps, yf)
    torch.cuda.synchronize()
    assert torch.equal(yf, sess.yf)
    st, word = cr.cr_get_device_status()
    assert st == cr.CR_OK, word
