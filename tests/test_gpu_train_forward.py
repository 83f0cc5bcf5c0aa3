"""The training update's forward is the serving forward: the y_f it leaves in its workspace
(for W_out's gradient) is what compress and forward give for the same weights, bit for bit,
also where scores far outgrow those of a row's first key tile."""
import numpy as np
import pytest
import torch

import fixtures as F
import oracle as O
from paper_2609_35139_gb300 import RepairSession, dims_from, pack_host_weights
from paper_2609_35139_gb300.session import Assembled
from test_gpu_train import _batch, _session, _step, lib  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("scale", [1.0, 6.0])
@pytest.mark.parametrize("mask", ["block_causal", "block_diagonal"])
def test_training_forward_is_the_serving_forward(mask, scale):
    case = F.make_case("small_multi", repairer=F.RepairerDims(8, 128, 256, 2, 8, 1024),
                       requests=[[2, 6, 0, 5], [6], [0, 3, 2, 6, 1]])
    d_b = 256
    for b in range(2):
        w = O.dtype_to_f64(case.weights[f"blk{b}.w_qkv"], "bf16")
        w[:2 * d_b] *= scale
        case.weights[f"blk{b}.w_qkv"] = F.f32_to_bf16(w.astype(np.float32))
    a = _batch(case)
    ts, dev, n = _session(case, a)
    _step(ts, dev, a, n, 0.0, mask)

    t, r = dims_from(case.target, case.repairer)
    sess = RepairSession(t, r, pack_host_weights(case.weights, 2), n)
    for dst, src in ((sess.kv, "kv"), (sess.emb, "emb"), (sess.chunk_end, "ce"), (sess.pos, "pos")):
        dst.copy_(dev[src])
    whole = Assembled(n, np.asarray(a["cu_seqlens"], np.int32))
    sess.compress(whole)
    sess.forward(whole, mask_mode=mask)
    torch.cuda.synchronize()
    want = sess.yf.reshape(-1).view(torch.int16)
    # (the workspace's parts start on 256-byte lines)
    ws = ts.workspace[:ts.workspace.numel() // 256 * 256].view(torch.int16)
    lines = ws.view(-1, 128)
    at = (lines == want[:128]).all(1).nonzero().flatten().tolist()
    assert any(torch.equal(ws[128 * k:128 * k + want.numel()], want) for k in at)
