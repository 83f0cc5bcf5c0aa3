"""Band walks of the GEMM where they run for certain: the width and band rules restated here
say that a call takes 256-wide tiles in bands, and its bits are those of the same rows in
calls small enough for one band.  Linears, QKV with RoPE, the three bf16 heads and the
encoder's two-product launch."""
import numpy as np
import pytest
import torch

from paper_2609_35139_gb300 import RepairSession, cr
from paper_2609_35139_gb300.session import Assembled

pytestmark = pytest.mark.gpu


def _ceil(a, b):
    return -(-a // b)


def _width(M, N):
    """The bf16 and plain fp32 epilogues' tile width: least rounds x (256 + width), wider on ties."""
    pairs = torch.cuda.get_device_properties(0).multi_processor_count // 2
    return min((256, 192, 128), key=lambda w: (_ceil(_ceil(M, 256) * _ceil(N, w), pairs) * (256 + w), -w))


def _band(M, N, K, terms=1, line=64e6, size=20e6):
    """Row tiles per band, 0 for one band."""
    if M * K * 2 * terms <= line or N <= 256:
        return 0
    if N * K * 2 <= 10e6:
        return 1
    band = max(1, int(size / (256 * K * 2 * terms)))
    return 0 if band >= _ceil(M, 256) else band


def _gen(seed):
    g = torch.Generator("cuda").manual_seed(seed)
    return lambda *s: torch.randn(s, generator=g, device="cuda")


# one row tile a band, and several with a last band that is not full
@pytest.mark.parametrize("M,N,K,rows", [(17001, 512, 2048, 1), (8700, 1520, 4096, 9), (5300, 3056, 6664, 5)])
@pytest.mark.parametrize("epi", [cr.CR_EPI_BF16, cr.CR_EPI_GELU_BF16, cr.CR_EPI_ADD_F32, cr.CR_EPI_F32])
def test_linears(epi, M, N, K, rows):
    assert _band(M, N, K) == rows and (epi == cr.CR_EPI_ADD_F32 or _width(M, N) == 256)
    assert rows == 1 or _ceil(M, 256) % rows
    rand = _gen(M)
    A, W, b = rand(M, K).to(torch.bfloat16), (rand(N, K) / K ** 0.5).to(torch.bfloat16), rand(N)
    f32 = epi in (cr.CR_EPI_ADD_F32, cr.CR_EPI_F32)
    whole = rand(M, N) if f32 else torch.empty(M, N, dtype=torch.bfloat16, device="cuda")
    parts = whole.clone()
    cr.cr_linear(A, W, b, whole, epi)
    for r in range(0, M, 1024):
        cr.cr_linear(A[r:r + 1024], W, b, parts[r:r + 1024], epi)
    torch.cuda.synchronize()
    assert torch.equal(whole, parts)


def test_qkv_rope():
    M, db, nh = 32001, 1024, 16
    assert _band(M, 3 * db, db) == 1 and _width(M, 3 * db) == 256
    rand = _gen(1)
    u, w, b = rand(M, db).to(torch.bfloat16), (rand(3 * db, db) / 32).to(torch.bfloat16), rand(3 * db)
    pos = torch.arange(M, dtype=torch.int32, device="cuda") % 5000
    whole, parts = (torch.empty(M, 3 * db, dtype=torch.bfloat16, device="cuda") for _ in range(2))
    cr.cr_qkv_rope(u, w, b, pos, db, nh, 1e4, whole)
    for r in range(0, M, 4096):
        cr.cr_qkv_rope(u[r:r + 4096], w, b, pos[r:r + 4096], db, nh, 1e4, parts[r:r + 4096])
    torch.cuda.synchronize()
    assert torch.equal(whole, parts)


@pytest.mark.parametrize("layers,rope,rows", [(2, False, 1), (2, True, 1), (4, False, 26), (4, True, 38)])
def test_heads(layers, rope, rows):
    """The in-place head in short calls against the in-place, pool and paged head in one."""
    heads, dh, db, lens = 8, 128, 1024, [9000, 7777, 16001, 679]
    n, D = sum(lens), 2 * layers * heads * dh
    assert _band(n, D, db, size=20e6 if rope else 14e6) == rows and (rows == 1 or _ceil(n, 256) % rows)
    rand = _gen(layers)
    w = {"w_out": (rand(D, db) / 32).to(torch.bfloat16), "b_out": rand(D), "sigma_stale": rand(D).abs() + 0.5,
         "sigma_delta": rand(D).abs() + 0.5}
    t = cr.target_dims(layers, heads, dh, 128, "bf16")
    r = cr.repairer_dims(8, 64, db, 0, 16, 256, 1e-5, 1e4)
    sess = RepairSession(t, r, cr.PackedWeights(w, 0), n)
    stale = rand(n, D).to(torch.bfloat16)
    sess.kv.copy_(stale)
    sess.yf.copy_(rand(n, db))
    sess.pos.copy_(torch.arange(n, dtype=torch.int32, device="cuda"))
    inv = (1e6 ** (-2.0 * np.arange(dh // 2) / dh)).astype(np.float32) if rope else None
    mode = cr.CR_ROPE_GLOBAL if rope else cr.CR_ROPE_NONE
    want = stale.clone()
    for a in range(0, n, 4096):
        m = min(4096, n - a)
        cr.cr_apply_residual(t, r, sess.weights, sess.yf[a:a + m], m, want[a:a + m], sess.pos[a:a + m], inv, mode,
                             workspace=sess.workspace)
    whole = Assembled(n, np.asarray([0, n], np.int32))

    slots = np.random.default_rng(1).permutation(n + 7)[:n].astype(np.int64)
    paged = torch.zeros((2 * layers, n + 7, heads * dh), dtype=torch.bfloat16, device="cuda")
    sess.apply_paged(whole, torch.from_numpy(slots).cuda(), paged, n + 7, inv, mode)
    torch.cuda.synchronize()
    assert torch.equal(paged[:, slots].transpose(0, 1).reshape(n, D), want)
    assert torch.equal(sess.kv, stale)

    sess.apply(whole, inv, mode)
    torch.cuda.synchronize()
    assert torch.equal(sess.kv, want)

    # the pool holds the request's rows as chunks, in another order
    order, at = [2, 0, 3, 1], np.concatenate([[0], np.cumsum(lens)])
    pool = torch.cat([stale[at[k]:at[k + 1]] for k in order])
    chunk_len = np.asarray([lens[k] for k in order], np.int32)
    chunk_start = np.concatenate([[0], np.cumsum(chunk_len)[:-1]]).astype(np.int64)
    sess.kv.zero_()
    sess.apply_pool(whole, pool, chunk_start, chunk_len, np.argsort(order).astype(np.int32),
                    np.asarray([0, 4], np.int32), inv, mode)
    torch.cuda.synchronize()
    assert torch.equal(sess.kv, want)


# W of the first pair below and above 10 MB
@pytest.mark.parametrize("dc,dm,rows", [(256, 2048, 1), (1024, 4096, 4)])
def test_encoder_products(dc, dm, rows):
    layers, heads, dh, db = 2, 8, 128, 256
    n = int(128e6 / (4 * dm)) + 701
    S = 2 * layers * heads
    assert _band(n, 2 * dc, max(dm, S * 8), 2, 128e6) == rows and (rows == 1 or _ceil(n, 256) % rows)
    rand = _gen(dc)
    mat = lambda o, i: (rand(o, i) / i ** 0.5).to(torch.bfloat16)  # noqa: E731
    w = {"w_seg": (rand(S, 8, dh) / 11).to(torch.bfloat16), "b_seg": rand(S, 8), "w_map": mat(dc, S * 8), "b_map": rand(dc),
         "w_tok": mat(dc, dm), "b_tok": rand(dc), "w_fuse": mat(db, 2 * dc), "b_fuse": rand(db), "w_rein": mat(db, dc)[None],
         "b_rein": rand(1, db), "sigma_stale": rand(S * dh).abs() + 0.5, "sigma_delta": rand(S * dh).abs() + 0.5}
    for k, o, i in (("qkv", 3 * db, db), ("o", db, db), ("fc1", 256, db), ("fc2", db, 256)):   # not run
        w[f"blk0.w_{k}"], w[f"blk0.b_{k}"] = mat(o, i), rand(o)
    for k in ("blk0.ln1", "blk0.ln2", "lnf"):
        w[f"{k}_g"], w[f"{k}_b"] = rand(db), rand(db)
    t = cr.target_dims(layers, heads, dh, dm, "bf16")
    r = cr.repairer_dims(8, dc, db, 1, 4, 256, 1e-5, 1e4)
    sess = RepairSession(t, r, cr.PackedWeights(w, 1), n)
    sess.kv.copy_(rand(n, S * dh))
    sess.emb.copy_(rand(n, dm))
    sess.compress(Assembled(n, np.asarray([0, n], np.int32)))
    h0, rein = torch.empty_like(sess.h0), torch.empty_like(sess.rein)
    for a in range(0, n, 2048):
        m = min(2048, n - a)
        cr.cr_compress_features(t, r, sess.weights, sess.kv[a:a + m], sess.emb[a:a + m], m, h0[a:a + m], rein[a:a + m],
                                sess.workspace)
        torch.cuda.synchronize()
    assert torch.equal(sess.h0, h0) and torch.equal(sess.rein, rein)
