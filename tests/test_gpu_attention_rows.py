"""Attention rows at the limits of their arithmetic: many small weights under a large one, values
that leave no room above them, one weight that is all of the sum."""
import numpy as np
import pytest
import torch

import fixtures as F
import oracle as O
from paper_2609_35139_gb300 import cr
from parity_util import as_f64, to_dev, to_host

pytestmark = pytest.mark.gpu


def _call(qkv, db, nh, n):
    out = torch.full((n, db), float("nan"), dtype=torch.bfloat16, device="cuda")
    end = torch.full((n,), n, dtype=torch.int32, device="cuda")
    cr.cr_masked_attention(qkv, db, nh, "bidirectional", end, torch.zeros_like(end), np.array([0, n], np.int32), out)
    torch.cuda.synchronize()
    st, word = cr.cr_get_device_status()
    assert st == cr.CR_OK, word
    return out


@pytest.mark.parametrize("nh,hd,q0,k0", [(2, 64, 8.0, 16.875), (4, 32, 4.0, 23.875)])
def test_small_weights_under_a_large_one(nh, hd, q0, k0):
    """One key of weight 1 with V = 1, 262143 keys of weight e^-16.9 (0.39 of the last bit of
    1 in fp32) with V = 0: every output is 1 / (1 + the sum of the small weights).  A sum
    that adds them to the large one by one drops them and is 0.6 % or more too small."""
    n, db = 262144, nh * hd
    qkv = torch.zeros((n, 3, nh, hd), dtype=torch.bfloat16, device="cuda")
    qkv[:, 0, :, 0] = q0
    qkv[0, 1, :, 0] = k0
    qkv[0, 2] = 1.0
    small = (n - 1) * float(np.exp(-q0 * k0 / np.sqrt(hd)))
    want = 1.0 / (1.0 + small)
    got = _call(qkv.reshape(n, 3 * db), db, nh, n).double()
    # half a bf16 step below 1, and 1 % of the small weights' part: a tile's 128 of them come
    # to 50 last bits of 1, of which each tile's addition may round half a bit
    bound = 2.0 ** -9 + 0.01 * small
    assert float((got - want).abs().max()) <= bound, (float(got.min()), float(got.max()), want)


@pytest.mark.parametrize("step", [0, 20, 50])
@pytest.mark.parametrize("hd", [64, 32])
def test_huge_values(hd, step):
    """Values of 2^100 with scores that outgrow the first key tile by about 2^step: the sums
    before the division pass fp32's range unless the reference follows, the outputs do not."""
    g = np.random.default_rng(hd + step)
    nh, n = 4, 700
    db = nh * hd
    x = g.standard_normal((n, 3, db)).astype(np.float32)
    x[128:, 1] *= max(1.0, step / 3 / np.log2(np.e))
    x[:, 2] *= 2.0 ** 100
    qkv = F.f32_to_bf16(x.reshape(n, 3 * db))
    got, q = as_f64(to_host(_call(to_dev(qkv), db, nh, n))), as_f64(qkv)
    part = lambda i: q[:, i * db:(i + 1) * db].reshape(n, nh, hd)
    m = O.attention_mask(np.zeros(n, np.int32), "bidirectional")
    want = O.masked_attention(part(0), part(1), part(2), m).reshape(n, db)
    mag = O.masked_attention(part(0), part(1), np.abs(part(2)), m).reshape(n, db)
    smax = np.abs(np.einsum("ihd,jhd->hij", part(0), part(1))).max() / np.sqrt(hd) * np.log2(np.e)
    # P and the output rounded to bf16 (2^-9 each, 2x margin), and the fp32 score and its
    # scaled difference: a few 2^-24 of the largest score in the exponent
    bound = 2.0 ** -8 * (mag + np.abs(want)) + 2.0 ** -20 * smax * mag
    assert np.isfinite(got).all()
    assert float((np.abs(got - want) / bound).max()) <= 1.0


@pytest.mark.parametrize("key", [5, 200, 699])
@pytest.mark.parametrize("nh,hd", [(2, 64), (4, 32)])
def test_one_key_takes_all(nh, hd, key):
    """One key outweighs all others by 2^46 to 2^57, another factor in each row: the
    row is that key's value exactly, as its weight is 1, which bf16 holds.  A reference below
    the row's maximum would round it."""
    n, db = 700, nh * hd
    g = torch.Generator("cuda").manual_seed(key)
    qkv = torch.zeros((n, 3, nh, hd), dtype=torch.bfloat16, device="cuda")
    qkv[:, 0, :, 0] = 16 + torch.rand((n, nh), generator=g, device="cuda") * 3.5
    qkv[key, 1, :, 0] = 2.0 * hd ** 0.5
    qkv[:, 2] = torch.randn((n, nh, hd), generator=g, device="cuda").to(torch.bfloat16)
    want = qkv[key, 2].reshape(1, db).expand(n, db).clone()
    assert torch.equal(_call(qkv.reshape(n, 3 * db), db, nh, n), want)
