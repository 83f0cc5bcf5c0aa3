"""A training update large enough that every warp of the LayerNorm backward takes several
rows and every attention CTA of the forward several items, over ragged requests, against
the oracle tensor by tensor.  The gradient buffer starts as NaN: each tensor is written
whole, and nothing is added to what was there."""
import numpy as np
import pytest
import torch

import fixtures as F
import oracle as O
from oracle import training as T
from paper_2609_35139_gb300 import cr
from test_gpu_train import _batch, _session, _step, _tensor, lib  # noqa: F401

pytestmark = pytest.mark.gpu

# pool chunks of 130, 77, 200, 1, 95, 64, 300 and 33 tokens
REQUESTS = [[0, 1, 2, 5], [6, 2], [7, 3, 0, 5, 6], [2, 6, 4], [6, 0, 3], [1, 2, 0], [4, 5, 6], [2, 0, 4], [6, 7, 2],
            [5, 2, 0, 1, 6], [3, 6, 4, 7], [2, 1, 6]]


@pytest.mark.parametrize("d_b,mask", [(256, "block_causal"), (512, "block_diagonal")])   # 8 heads of 32, of 64
def test_update_of_many_rows(d_b, mask):
    case = F.make_case("small_multi", repairer=F.RepairerDims(8, 128, d_b, 2, 8, 1024), requests=REQUESTS)
    a = _batch(case)
    t, r = case.target, case.repairer
    lens = np.diff(a["cu_seqlens"])
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    assert len(a["kv"]) > 3 * 8 * 148 and 8 * int(np.sum(-(-lens // 256))) > sms
    names = T.trained_names(r.n_blocks)
    params = {k: (O.dtype_to_f64(case.weights[k], "bf16") if case.weights[k].dtype == np.uint16
                  else case.weights[k].astype(np.float64)) for k in names}
    zeros = {k: np.zeros_like(v) for k, v in params.items()}
    loss, norm, grads, _, _, _ = T.train_step(params, zeros, zeros, 1, 1e-3, a, sigma_stale=case.weights["sigma_stale"],
                                              sigma_delta=case.weights["sigma_delta"], cache_dtype="bf16",
                                              head_dim=t.head_dim, n_heads=r.n_heads, mask_mode=mask)
    ts, dev, n = _session(case, a)
    ts.grads.fill_(float("nan"))
    stats = _step(ts, dev, a, n, 1e-3, mask)
    assert abs(float(stats[0]) - loss) <= 1e-3 * loss
    assert abs(float(stats[1]) - norm) <= 5e-3 * norm
    assert bool(torch.isfinite(ts.grads).all())
    # eight bf16 roundings of a GEMM operand (2^-9 each) in RMS, as in the small cases
    for k in names:
        gg, ref = _tensor(ts, ts.grads, k, params[k].shape), grads[k]
        cos = float((gg * ref).sum() / np.sqrt((gg ** 2).sum() * (ref ** 2).sum()))
        rel = float(np.sqrt(np.mean((gg - ref) ** 2)) / np.sqrt(np.mean(ref ** 2)))
        assert cos >= 0.9999 and rel <= 1.5e-2, (k, cos, rel)
    st, word = cr.cr_get_device_status()
    assert st == cr.CR_OK, word
