"""The attention kernel takes a row's softmax reference from its first visible key
tile and starts a CTA again where later scores outgrow it: scores that grow along the
keys by less and by far more than the restart limit (2^60), against the oracle."""
import numpy as np
import pytest
import torch

import fixtures as F
import oracle as O
from paper_2609_35139_gb300 import cr
from parity_util import as_f64, to_dev, to_host
from test_gpu_masks import MODES, _maps

pytestmark = pytest.mark.gpu

# one tile, a ragged map whose later chunks outgrow the first tile, several requests
GROWING = [[[90]], [[130, 300, 77]], [[260, 5], [1], [40, 700]]]


@pytest.mark.parametrize("step", [20, 55, 90, 1000])
@pytest.mark.parametrize("mode", MODES)
@pytest.mark.parametrize("reqs", GROWING)
@pytest.mark.parametrize("hd", [64, 32])
def test_growing_scores(hd, reqs, mode, step):
    """Keys after the first 128 of a request are scaled so that their scores (log2 units)
    have standard deviation step / 3: the largest exceed the first tile's by about step."""
    g = np.random.default_rng(step + hd)
    nh, db = 2, 2 * hd
    cend, _, cids, cu = _maps(reqs)
    N = int(cu[-1])
    x = g.standard_normal((N, 3 * db)).astype(np.float32)
    for a, b in zip(cu[:-1], cu[1:]):
        x[a + 128:b, db:2 * db] *= step / 3 / np.log2(np.e)
    qkv = F.f32_to_bf16(x)
    out = torch.full((N, db), float("nan"), dtype=torch.bfloat16, device="cuda")
    ce, cs = to_dev(cend), torch.empty(N, dtype=torch.int32, device="cuda")
    cr.cr_chunk_starts(ce, cu, N, cs)
    cr.cr_masked_attention(to_dev(qkv), db, nh, mode, ce, cs, cu, out)
    torch.cuda.synchronize()
    st, word = cr.cr_get_device_status()
    assert st == cr.CR_OK, word
    got, q = as_f64(to_host(out)), as_f64(qkv)
    for r in range(len(reqs)):
        a, b = cu[r], cu[r + 1]
        sl = lambda off: q[a:b, off:off + db].reshape(b - a, nh, hd)
        m = O.attention_mask(cids[r], mode)
        want = O.masked_attention(sl(0), sl(db), sl(2 * db), m).reshape(b - a, db)
        mag = O.masked_attention(sl(0), sl(db), np.abs(sl(2 * db)), m).reshape(b - a, db)
        smax = np.abs(np.einsum("ihd,jhd->hij", sl(0), sl(db))).max() / np.sqrt(hd) * np.log2(np.e)
        # P and the output rounded to bf16 (2^-9 each, 2x margin), and the fp32 score
        # and its scaled difference: a few 2^-24 of the largest score in the exponent
        bound = 2.0 ** -8 * (mag + np.abs(want)) + 2.0 ** -20 * smax * mag + 1e-5
        worst = float((np.abs(got[a:b] - want) / bound).max())
        assert worst <= 1.0, f"{mode} hd={hd} step={step} request {r}: error / bound = {worst:.3f}"


@pytest.mark.parametrize("mode", ["block_causal", "block_diagonal"])
@pytest.mark.parametrize("hd", [64, 32])
def test_more_items_than_sms(hd, mode):
    """Enough (request, head, query-tile pair) items that every CTA runs several, of one
    and of two query tiles; the scores of every seventh request outgrow the restart limit,
    so that some CTAs run items again after others."""
    g = np.random.default_rng(hd)
    nh, db = 8, 8 * hd
    reqs = [[int(x) for x in g.integers(1, 200, size=g.integers(1, 5))] for _ in range(90)]
    cend, _, cids, cu = _maps(reqs)
    N = int(cu[-1])
    x = g.standard_normal((N, 3 * db)).astype(np.float32)
    for r in range(0, len(reqs), 7):
        x[cu[r] + 128:cu[r + 1], db:2 * db] *= 70.0
    qkv = F.f32_to_bf16(x)
    out = torch.full((N, db), float("nan"), dtype=torch.bfloat16, device="cuda")
    ce, cs = to_dev(cend), torch.empty(N, dtype=torch.int32, device="cuda")
    cr.cr_chunk_starts(ce, cu, N, cs)
    cr.cr_masked_attention(to_dev(qkv), db, nh, mode, ce, cs, cu, out)
    torch.cuda.synchronize()
    st, word = cr.cr_get_device_status()
    assert st == cr.CR_OK, word
    got, q = as_f64(to_host(out)), as_f64(qkv)
    for r in range(len(reqs)):
        a, b = cu[r], cu[r + 1]
        sl = lambda off: q[a:b, off:off + db].reshape(b - a, nh, hd)
        m = O.attention_mask(cids[r], mode)
        want = O.masked_attention(sl(0), sl(db), sl(2 * db), m).reshape(b - a, db)
        mag = O.masked_attention(sl(0), sl(db), np.abs(sl(2 * db)), m).reshape(b - a, db)
        smax = np.abs(np.einsum("ihd,jhd->hij", sl(0), sl(db))).max() / np.sqrt(hd) * np.log2(np.e)
        bound = 2.0 ** -8 * (mag + np.abs(want)) + 2.0 ** -20 * smax * mag + 1e-5   # as above
        worst = float((np.abs(got[a:b] - want) / bound).max())
        assert worst <= 1.0, f"{mode} hd={hd} request {r} {reqs[r]}: error / bound = {worst:.3f}"
