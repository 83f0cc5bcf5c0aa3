"""Attention where something is wrong outside it: a chunk map that no host check sees, a
wait of an earlier kernel that gave up.  Nothing here faults or hangs a GPU; every wait in
the kernel is bounded."""
import numpy as np
import pytest
import torch

import fixtures as F
from paper_2609_35139_gb300 import cr
from parity_util import to_dev
from test_gpu_masks import _maps

pytestmark = pytest.mark.gpu


def _call(qkv, db, nh, mode, cend, cstart, cu):
    out = torch.full((int(cu[-1]), db), float("nan"), dtype=torch.bfloat16, device="cuda")
    cr.cr_masked_attention(qkv, db, nh, mode, to_dev(cend), to_dev(cstart), cu, out)
    torch.cuda.synchronize()
    return out


@pytest.mark.parametrize("tile", ["first", "second", "both"])
@pytest.mark.parametrize("mode", ["block_causal", "block_diagonal"])
def test_keys_that_end_before_the_first_key_tile(mode, tile):
    """A malformed map that ends a query tile's keys before its pair's first key tile: the
    tile has no key tiles, and every other request's rows stay what they are.  Enough
    items that CTAs run several, so that a ring out of step would show in the next one."""
    g = np.random.default_rng(3)
    nh, hd = 16, 64
    db = nh * hd
    reqs = [[int(x) for x in g.integers(100, 400, size=2)] for _ in range(16)]
    cend, cstart, _, cu = _maps(reqs)
    qkv = to_dev(F.f32_to_bf16(g.standard_normal((int(cu[-1]), 3 * db)).astype(np.float32)))
    want = _call(qkv, db, nh, mode, cend, cstart, cu)
    bad = list(range(1, len(reqs), 3))
    for r in bad:
        a, b = int(cu[r]), int(cu[r + 1])
        if tile != "second":
            cend[a + 127] = -1000
        if tile != "first":
            cend[a + min(255, b - a - 1)] = -1000
    got = _call(qkv, db, nh, mode, cend, cstart, cu)
    st, word = cr.cr_get_device_status()
    assert st == cr.CR_OK, word
    for r in range(len(reqs)):
        if r not in bad:
            assert torch.equal(got[cu[r]:cu[r + 1]], want[cu[r]:cu[r + 1]]), f"request {r}"


@pytest.mark.parametrize("mode", ["block_causal", "block_diagonal"])
@pytest.mark.parametrize("hd", [64, 32])
def test_attention_after_a_wait_gave_up(hd, mode):
    """A kernel before has given up, so this call's waits may give up, too, at any point:
    the call ends by itself with its copies landed, and once the status is cleared the
    same call is right again."""
    g = np.random.default_rng(hd)
    nh, reqs = 8, [[int(x) for x in g.integers(100, 400, size=3)] for _ in range(20)]
    db = nh * hd
    cend, cstart, _, cu = _maps(reqs)
    qkv = to_dev(F.f32_to_bf16(g.standard_normal((int(cu[-1]), 3 * db)).astype(np.float32)))
    want = _call(qkv, db, nh, mode, cend, cstart, cu)
    assert cr.cr_get_device_status()[0] == cr.CR_OK
    try:
        cr.cr_wait_selftest()
        for _ in range(4):
            _call(qkv, db, nh, mode, cend, cstart, cu)
        assert cr.cr_get_device_status()[0] == cr.CR_ERR_TIMEOUT
    finally:
        cr.cr_clear_device_status()
    for _ in range(4):
        assert torch.equal(_call(qkv, db, nh, mode, cend, cstart, cu), want)
    assert cr.cr_get_device_status()[0] == cr.CR_OK
