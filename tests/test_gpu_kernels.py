"""Kernel variants and dispatch rules at the sizes where they change: edges of tiles, remainders, the ends of a range.
Every comparison is bit for bit against the oracle."""
import numpy as np
import pytest

import oracle
import synth
from gpu_util import assert_same_bits, dev, empty, host, ws

pytestmark = pytest.mark.gpu
F = np.float32


@pytest.fixture(scope="module")
def det():
    import paper_2609_17380_b200 as d
    d.load()
    return d


def _sync():
    import torch
    torch.cuda.synchronize()


# chunk counts of a launch around the rule between the two hash kernels (a warp of eight chains per scheduler: 8 * 4 * SMs),
# between one and two warps per eight chains (half of that) and between plain and multiply-add additions (a warp of 32 chunks per
# scheduler), byte counts around every place that the padding of a block can start at,
# tensors of one, two and three levels, an empty one, byte counts off the 4- and 64-byte grid, more tensors than one
# launch takes
@pytest.mark.parametrize("sizes", [
    [16, 0, 4096, 4095, 4097, 61, 64, 55, 56, 128 * 4096, 128 * 4096 + 1, 0],
    "edge", "edge+1", "pair", "pair+1", "flat", "flat+1", list(range(1, 130)) + [4096 + i for i in range(1, 65)], [128 * 128 * 4096 + 4096 + 48, 5000, 129 * 4096 + 3],
    [(37 * i) % 9000 for i in range(300)],
])
def test_hash_batch(det, sizes):
    if isinstance(sizes, str):
        edge = {"edge": 32, "pair": 16, "flat": 128}[sizes.split("+")[0]] * det.det_device_sm_count()
        sizes = [4096 * (edge - 200) + 4096 * sizes.endswith("+1"), 4096 * 199 + 777]          # edge or edge + 1 chunks
    rng = np.random.default_rng(len(sizes))
    blobs = [rng.integers(0, 256, n).astype(np.uint8) for n in sizes]
    tensors = [dev(b) for b in blobs]
    roots = empty((32 * len(sizes),), np.uint8)
    det.det_tensor_hash_batch(tensors, roots, ws(det.det_tensor_hash_batch_ws_bytes(tensors)))
    _sync()
    raw = host(roots).tobytes()
    for i, b in enumerate(blobs):
        assert raw[32 * i:32 * i + 32].hex() == oracle.tensor_hash(b), (i, sizes[i])


# LM head through its entry points, ragged rows and columns; at these sizes the dispatch takes 32x64 and 128x128 tiles (every tile is run by
# test_lmhead_every_tile); the last one has a grid of several full rounds in the weight gradient
@pytest.mark.parametrize("M,V,K", [(8, 16, 16), (40, 80, 48), (136, 2064, 80), (392, 4112, 176), (1032, 8208, 32), (264, 16400, 528)])
def test_lmhead_tiles(det, M, V, K):
    H, W = synth.normal_bf16((M, K), 1.0, seed=M, tid=1), synth.normal_bf16((V, K), 0.05, seed=M, tid=2)
    lg = empty((M, V), F)
    det.det_lmhead_fwd(dev(H), dev(W), M, V, K, lg)
    _sync()
    assert_same_bits(host(lg), oracle.lmhead_fwd(H, W), "logits")
    g = synth.normal_f32((M, V), 1e-3, seed=M, tid=3)
    dH, dW = empty((M, K), np.uint16), empty((V, K), F)
    det.det_lmhead_bwd(dev(g), dev(H), dev(W), M, V, K, dH, dW, 1)
    _sync()
    dH_o, dW_o = oracle.lmhead_bwd(g, H, W)
    assert_same_bits(host(dH, np.uint16), dH_o, "dH")
    assert_same_bits(host(dW), dW_o, "dW")


# the three contractions of the head on each of the four tiles: one tile and less, ragged rows and columns in the last tile of either
# direction, one slab and many, a weight gradient that goes on from a chunk before, slabs with values whose products can be subnormal
@pytest.mark.parametrize("tile", [0, 1, 2, 3])
@pytest.mark.parametrize("M,V,K,tiny", [(8, 16, 16, False), (136, 272, 304, False), (200, 528, 80, True), (392, 784, 560, True)])
def test_lmhead_every_tile(det, tile, M, V, K, tiny):
    H, W = synth.normal_bf16((M, K), 1.0, seed=M, tid=1), synth.normal_bf16((V, K), 0.05, seed=M, tid=2)
    g = synth.normal_f32((M, V), 1e-3, seed=M, tid=3)
    if tiny:
        rng = np.random.default_rng(M)
        for a in (H, W, g):
            at = rng.integers(0, a.size, 12)
            v = (F(2.0) ** rng.integers(-66, -61, 12)).astype(F)
            a.reshape(-1)[at] = v if a is g else synth.to_bf16(v)
    dH_, dW_, dg = dev(H), dev(W), dev(g)
    lg, dH, dW = empty((M, V), F), empty((M, K), np.uint16), empty((V, K), F)
    det.det_test_lmhead_tile(0, tile, dH_, dW_, M, V, K, lg)
    det.det_test_lmhead_tile(1, tile, dg, dW_, M, V, K, dH)
    det.det_test_lmhead_tile(2, tile, dg, dH_, M, V, K, dW, 1)
    _sync()
    dH_o, dW_o = oracle.lmhead_bwd(g, H, W)
    assert_same_bits(host(lg), oracle.lmhead_fwd(H, W), "logits")
    assert_same_bits(host(dH, np.uint16), dH_o, "dH")
    assert_same_bits(host(dW), dW_o, "dW")
    det.det_test_lmhead_tile(2, tile, dg, dH_, M, V, K, dW, 0)
    _sync()
    assert_same_bits(host(dW), oracle.lmhead_bwd(g, H, W, dW_o)[1], "dW continued")


# contraction lengths around a ring slot of two, three and four slabs of 16 and around the ring's two slots, the last slab of the weight gradient a
# half one or whole; rows of which the last tile repeats most
@pytest.mark.parametrize("tile", [0, 1, 2, 3])
@pytest.mark.parametrize("C", [32, 48, 64, 80, 96, 112, 128, 144])
def test_lmhead_slots_of_slabs(det, tile, C):
    H, W = synth.normal_bf16((24, C), 1.0, seed=C, tid=1), synth.normal_bf16((C, C), 0.05, seed=C, tid=2)
    g = synth.normal_f32((24, C), 1e-3, seed=C, tid=3)
    lg, dH = empty((24, C), F), empty((24, C), np.uint16)
    det.det_test_lmhead_tile(0, tile, dev(H), dev(W), 24, C, C, lg)
    det.det_test_lmhead_tile(1, tile, dev(g), dev(W), 24, C, C, dH)
    _sync()
    assert_same_bits(host(lg), oracle.lmhead_fwd(H, W), "logits")
    assert_same_bits(host(dH, np.uint16), oracle.lmhead_bwd(g, H, W)[0], "dH")
    for M in (C - 8, C):
        Hm, gm = synth.normal_bf16((M, 16), 1.0, seed=M, tid=4), synth.normal_f32((M, 32), 1e-3, seed=M, tid=5)
        dW = empty((32, 16), F)
        det.det_test_lmhead_tile(2, tile, dev(gm), dev(Hm), M, 32, 16, dW, 1)
        _sync()
        assert_same_bits(host(dW), oracle.lmhead_bwd(gm, Hm, synth.normal_bf16((32, 16), 0.05, seed=M, tid=6))[1], "dW")


# the tile that the head's forward takes at sizes where the rates of strided operands would choose a slower one
@pytest.mark.parametrize("M,V,K,tile", [(640, 2048, 640, 1), (640, 2048, 2048, 1), (832, 16384, 2048, 1), (304, 37424, 1408, 0), (88, 14128, 496, 1), (384, 2048, 2048, 2)])
def test_lmhead_forward_tile(det, M, V, K, tile):
    if det.det_device_sm_count() != 148:
        pytest.skip("measured on 148 SMs")
    assert det.det_test_lmhead_pick(M, V, K) == tile


# version-2 gradients where a row of logits is long enough for eight warps (4096 values), and one step below; a token gradient of 36
# tiles and 16 steps (two CTAs a tile, bf16 results), one of 80 (pairs, bf16 results); the 1B shape's vocabulary, an odd number of row
# tiles for the weight gradient
@pytest.mark.parametrize("M,V,K", [(128, 3968, 128), (128, 4096, 128), (256, 8320, 128), (1152, 2048, 512), (1280, 2048, 1024),
                                   (256, 50304, 128)])
def test_lmhead_v2_long_rows(det, M, V, K):
    import torch
    from oracle import v2
    H, W = synth.normal_bf16((M, K), 1.0, seed=V, tid=1), synth.normal_bf16((V, K), 0.05, seed=V, tid=2)
    g = synth.normal_f32((M, V), 1e-3, seed=V, tid=3)
    g[5, V - 1] = np.inf                                          # seen by one warp: its row of dH and its row of dW are NaN
    dH, dW = empty((M, K), np.uint16), empty((V, K), F)
    status = torch.zeros(1, dtype=torch.int32, device="cuda")
    det.det_lmhead_bwd_v2(dev(g), dev(H), dev(W), M, V, K, dH, dW, ws(det.det_lmhead_bwd_v2_ws_bytes(M, V, K)), status)
    _sync()
    assert int(status.item()) == 0
    want_H, want_W = v2.lmhead_bwd(g, H, W)
    got_H, got_W = host(dH, np.uint16), host(dW)
    assert np.isnan(synth.from_bf16(got_H[5])).all() and np.isnan(got_W[V - 1]).all()
    assert_same_bits(np.delete(got_H, 5, 0), np.delete(want_H, 5, 0), "version-2 dH")
    assert_same_bits(got_W[:-1], want_W[:-1], "version-2 dW")


# version-2 contraction on both sides of where the CTAs that share a tile change (15 and 16 steps; 32 steps with 32 and 33 tiles, 16
# with 74 and 75) and of where CTA pairs begin (one round of tiles with 14 and 15 steps, two with 7 and 8, three with 5 and 6), and
# operands whose exponents cross the range in which every result is a normal number, in both directions
@pytest.mark.parametrize("M,V,K,spread", [(128, 128, 1920, False), (128, 128, 2048, False), (256, 128, 4096, True), (128, 4224, 4096, False),
                                          (512, 1024, 4096, False), (256, 4736, 2048, False), (128, 9600, 2048, False),
                                          (256, 5120, 1792, False), (256, 5120, 1920, False), (256, 9728, 896, False), (256, 9728, 1024, False),
                                          (768, 6912, 640, False), (768, 6912, 768, True),
                                          (256, 384, 256, True), (256, 20480, 128, False), (768, 6912, 384, True)])
def test_lmhead_v2_shared_tiles(det, M, V, K, spread):
    import torch
    from oracle import v2
    H, W = synth.normal_bf16((M, K), 1.0, seed=V + K, tid=1), synth.normal_bf16((V, K), 0.05, seed=V + K, tid=2)
    if spread:                                                    # rows of H from 2^-70 to 2^70 times, blocks of W by 2^60 either way
        h = synth.from_bf16(H) * np.exp2(np.linspace(-70, 70, M).round())[:, None]
        w = synth.from_bf16(W) * np.exp2(60.0 * ((np.arange(V) // 64) % 3 - 1))[:, None]
        H, W = synth.to_bf16(h.astype(F)), synth.to_bf16(w.astype(F))
    lg = empty((M, V), F)
    status = torch.zeros(1, dtype=torch.int32, device="cuda")
    det.det_lmhead_fwd_v2(dev(H), dev(W), M, V, K, lg, ws(det.det_lmhead_fwd_v2_ws_bytes(M, V, K)), status)
    _sync()
    assert int(status.item()) == 0
    assert_same_bits(host(lg), v2.lmhead_fwd(H, W), "version-2 logits")


# the longest contraction that is allowed, with the largest slices (bf16 reaches 16320 of 16383): totals up to 2^43.99 of either sign, ties of
# the one rounding and their neighbours, accumulators that reach their largest, on each form of the contraction (four and two CTAs a tile,
# one, pairs).  Four kinds of rows and thirty-two of columns, so the oracle takes one of each
@pytest.mark.parametrize("M,V", [(128, 128), (128, 4224), (128, 9600), (256, 9728)])
def test_lmhead_v2_largest_totals(det, M, V):
    import torch
    from oracle import v2
    K, big = 65408, F(255.0 / 128)                                # 16320 = 255 * 64
    h, w = np.full((4, K), big, F), np.full((32, K), big, F)
    h[1], h[2, ::2], h[3] = -big, -big, F(1.0)                    # h[3]: products of 2^13, so that a column's sum is what is rounded
    for i in range(32):                                           # sums of 2^29.99 with a tail of 31 .. 33 of 64 (a tie at 32)
        w[i, 7 + i] = F((32 + 64 * (i % 4 // 2) + (i // 4) % 3 - 1) / 8192.0)
    w[1::2] *= F(-1.0)
    w[28:30, 0::3] = F(255.0 / 8192)                              # low slices of 127
    H, W = synth.to_bf16(h), synth.to_bf16(w)
    want = np.tile(v2.lmhead_fwd(H, W), (M // 4, V // 32))
    assert np.abs(want).max() > 65400 * 3.96
    lg = empty((M, V), F)
    status = torch.zeros(1, dtype=torch.int32, device="cuda")
    det.det_lmhead_fwd_v2(dev(H).repeat(M // 4, 1), dev(W).repeat(V // 32, 1), M, V, K, lg, ws(det.det_lmhead_fwd_v2_ws_bytes(M, V, K)), status)
    _sync()
    assert int(status.item()) == 0
    assert_same_bits(host(lg), want, "version-2 logits")


# rows that are all non-finite for one warp against columns of which one is: every one of its results is NaN, the others stay as they are
@pytest.mark.parametrize("M,V,K", [(128, 128, 128), (256, 9728, 1024)])
def test_lmhead_v2_non_finite_warp(det, M, V, K):
    import torch
    from oracle import v2
    H, W = synth.normal_bf16((M, K), 1.0, seed=M, tid=1), synth.normal_bf16((V, K), 0.05, seed=M, tid=2)
    H[32:64, 3] = synth.to_bf16(np.full(32, np.inf, F))
    H[40:44, 5] = synth.to_bf16(np.full(4, np.nan, F))
    W[70, 9] = synth.to_bf16(np.array([-np.inf], F))[0]
    lg = empty((M, V), F)
    status = torch.zeros(1, dtype=torch.int32, device="cuda")
    det.det_lmhead_fwd_v2(dev(H), dev(W), M, V, K, lg, ws(det.det_lmhead_fwd_v2_ws_bytes(M, V, K)), status)
    _sync()
    assert int(status.item()) == 0
    got, want = host(lg), v2.lmhead_fwd(H, W)
    bad = np.zeros((M, V), bool)
    bad[32:64], bad[:, 70] = True, True
    assert np.array_equal(np.isnan(got), bad) and np.array_equal(np.isnan(want), bad)
    assert_same_bits(got[~bad], want[~bad], "version-2 logits")


# attention with the form that the rule gives to the heads and rows (test_attention_forward_every_form runs each), S off the 128 grid, windows
# that start and end inside a block, grouped heads (one accumulator over the whole group)
@pytest.mark.parametrize("B,H,Hkv,S,W", [(1, 2, 2, 576, 0), (1, 40, 40, 320, 0), (2, 80, 80, 192, 0), (1, 3, 3, 704, 256),
                                         (1, 60, 60, 448, 128), (3, 64, 64, 320, 128), (1, 8, 2, 384, 0), (1, 6, 1, 448, 128)])
@pytest.mark.parametrize("fixq", [False, True])
def test_attention_row_blocks(det, B, H, Hkv, S, W, fixq):
    HD, KD = H * 128, Hkv * 128
    ld = HD + 2 * KD
    qkv = synth.normal_bf16((B * S, ld), 1.0, seed=S + H, tid=1)
    dout = synth.normal_bf16((B * S, HD), 0.1, seed=S + H, tid=2)
    x = dev(qkv)
    q = x.data_ptr()
    k, v = q + 2 * HD, q + 2 * (HD + KD)
    out, lse = empty((B * S, HD), np.uint16), empty((B, H, S), F)
    det.det_attn_fwd(q, k, v, ld, B, H, S, out, HD, lse, Hkv=Hkv, window=W)
    _sync()
    oout, olse = oracle.attn_fwd(qkv, B, H, S, Hkv=Hkv, window=W)
    assert_same_bits(host(lse), olse, "lse")
    assert_same_bits(host(out, np.uint16), oout, "out")
    dqkv = empty((B * S, ld), np.uint16)
    d = dqkv.data_ptr()
    bwd, need = (det.det_attn_bwd_fixq, det.det_attn_bwd_fixq_ws_bytes) if fixq else (det.det_attn_bwd, det.det_attn_bwd_ws_bytes)
    bwd(dev(dout), q, k, v, out, lse, ld, HD, B, H, S, d, d + 2 * HD, d + 2 * (HD + KD), ld, ws(need(B, H, S, Hkv)), Hkv=Hkv, window=W)
    _sync()
    want = oracle.attn_bwd(dout, qkv, oout, olse, B, H, S, Hkv=Hkv, window=W, fixq=fixq)
    got = host(dqkv, np.uint16)
    for name, lo, hi in (("dq", 0, HD), ("dk", HD, HD + KD), ("dv", HD + KD, ld)):
        assert_same_bits(got[:, lo:hi], want[:, lo:hi], name)


def _underflow(qkv, B, H, Hkv, S):
    """Values below 2^-63 whose products with factors that are not, subnormal, are what a sum shows that does not flush them.  In q and k: the
    first row of every head is seen by the first query alone, whose logsumexp is the logit itself, here 2^-116 and fifteen products of about
    2^-127; they lie in the 16 dimensions kvh mod 8.  In v: of dimension 10 + b all is zero but 16 keys of key block b, one 2^-115 and
    fifteen of 2^-125 .. 2^-126, which the weights bring below.  Zeros count as large, so a slab of 16 is the only one of its kind in a head."""
    rng = np.random.default_rng(S + H)
    HD, KD = H * 128, Hkv * 128
    x = synth.from_bf16(qkv).reshape(B, S, H + 2 * Hkv, 128).copy()
    q, k, v = x[:, :, :H], x[:, :, H:H + Hkv], x[:, :, H + Hkv:]
    for h in range(H):
        d = 16 * (h // (H // Hkv) % 8)
        q[:, 0, h] = 0
        q[:, 0, h, d:d + 16] = F(2.0 ** -62) * (1 + rng.integers(0, 4, 16) / 8)
        q[:, 0, h, d] = F(2.0 ** -60)
    for h in range(Hkv):
        d = 16 * (h % 8)
        k[:, 0, h, d:d + 16] = F(2.0 ** -65)
        k[:, 0, h, d] = F(2.0 ** -56)
        for b in range(S // 128 if S > 128 else 1):
            at = 128 * b + 16 * ((h + b) % min(8, S // 16))
            v[:, :, h, 10 + b] = 0
            v[:, at:at + 16, h, 10 + b] = F(2.0 ** -126) * (1 + rng.integers(0, 8, 16) / 8)
            v[:, at, h, 10 + b] = F(2.0 ** -115)
    return synth.to_bf16(x.reshape(B * S, HD + 2 * KD))


# every form of the forward (rows per CTA; 33: 32 rows and two groups) at sizes of one row block up to several, off the 128 grid, grouped heads,
# windows that begin inside a block, one to three key blocks long; ordinary, saturated and underflowing inputs
@pytest.mark.parametrize("rows", [128, 64, 32, 33])
@pytest.mark.parametrize("B,H,Hkv,S,W", [(1, 8, 8, 64, 0), (1, 16, 8, 448, 0), (2, 8, 8, 640, 0), (1, 8, 8, 448, 128), (1, 16, 8, 704, 256), (2, 8, 8, 576, 384)])
@pytest.mark.parametrize("kind", ["plain", "saturated", "underflow"])
def test_attention_forward_every_form(det, rows, B, H, Hkv, S, W, kind):
    HD, KD = H * 128, Hkv * 128
    ld = HD + 2 * KD
    qkv = synth.normal_bf16((B * S, ld), 1.0, seed=S + W, tid=1)
    if kind == "saturated":
        qkv[:, :HD] = synth.to_bf16(synth.from_bf16(qkv[:, :HD]) * F(40.0))          # logits of order +-400
    elif kind == "underflow":
        qkv = _underflow(qkv, B, H, Hkv, S)
    d = dev(qkv)
    q = d.data_ptr()
    s_q = np.array([0.02], F)
    out, lse, codes = empty((B * S, HD), np.uint16), empty((B, H, S), F), empty((B * S, HD), np.int8)
    det.det_test_attn_fwd(rows, q, q + 2 * HD, q + 2 * (HD + KD), ld, B, H, S, out, HD, lse, dev(s_q), codes, Hkv=Hkv, window=W)
    _sync()
    oout, olse = oracle.attn_fwd(qkv, B, H, S, Hkv=Hkv, window=W)
    if kind == "underflow":
        assert (olse[:, :, 0] != 0).all() and (np.abs(olse[:, :, 0]) < 2.0 ** -110).all()
    assert_same_bits(host(lse), olse, "lse")
    assert_same_bits(host(out, np.uint16), oout, "out")
    assert_same_bits(host(codes).reshape(-1), np.asarray(oracle.lsq_quantize(oout, s_q, False)).reshape(-1).view(np.int8), "codes")


# the same products in the logits of the form with int8 P.V
@pytest.mark.parametrize("B,H,Hkv,S,W", [(1, 8, 8, 192, 0), (1, 16, 8, 448, 128)])
def test_int8_pv_underflow(det, B, H, Hkv, S, W):
    import torch
    HD, KD = H * 128, Hkv * 128
    ld = HD + 2 * KD
    qkv = _underflow(synth.normal_bf16((B * S, ld), 1.0, seed=S, tid=1), B, H, Hkv, S)
    d = dev(qkv)
    q = d.data_ptr()
    out, lse, status = empty((B * S, HD), np.uint16), empty((B, H, S), F), torch.zeros(1, dtype=torch.int32, device="cuda")
    det.det_attn_fwd_int8pv(q, q + 2 * HD, q + 2 * (HD + KD), ld, B, H, S, out, HD, lse, status, Hkv=Hkv, window=W)
    _sync()
    assert int(status.item()) == 0
    oout, olse = oracle.attn_fwd(qkv, B, H, S, Hkv=Hkv, window=W, int8_pv=True)
    assert (olse[:, :, 0] != 0).all() and (np.abs(olse[:, :, 0]) < 2.0 ** -110).all()
    assert_same_bits(host(lse), olse, "lse")
    assert_same_bits(host(out, np.uint16), oout, "out")


# which form the forward takes, where it has been measured on this device's SMs: four windows shorter than the sequence, one that is not
@pytest.mark.parametrize("heads,S,W,rows", [(16, 2048, 128, 128), (16, 4096, 512, 64), (8, 512, 256, 33), (32, 512, 128, 128), (8, 512, 512, 33)])
def test_attention_forward_form(det, heads, S, W, rows):
    if det.det_device_sm_count() != 148:
        pytest.skip("measured on 148 SMs")
    assert det.det_test_attn_rows(heads, S, W) == rows


# the backward on either side of the number of blocks (seven quarters of the SMs) from which warps of their own form P and dS: heads of two
# and of three blocks, the latter with half a block at the end and a window
@pytest.mark.parametrize("per_head,S,W", [(3, 256, 0), (5, 320, 128)])
@pytest.mark.parametrize("more", [0, 1])
def test_attention_backward_epilogue_warps(det, per_head, S, W, more):
    B, H = 1, 7 * det.det_device_sm_count() // 4 // per_head + more
    HD = H * 128
    qkv, dout = synth.normal_bf16((S, 3 * HD), 1.0, seed=H, tid=1), synth.normal_bf16((S, HD), 0.1, seed=H, tid=2)
    x, d = dev(qkv), empty((S, 3 * HD), np.uint16)
    q, g = x.data_ptr(), d.data_ptr()
    out, lse = empty((S, HD), np.uint16), empty((B, H, S), F)
    det.det_attn_fwd(q, q + 2 * HD, q + 4 * HD, 3 * HD, B, H, S, out, HD, lse, window=W)
    det.det_attn_bwd(dev(dout), q, q + 2 * HD, q + 4 * HD, out, lse, 3 * HD, HD, B, H, S, g, g + 2 * HD, g + 4 * HD, 3 * HD,
                     ws(det.det_attn_bwd_ws_bytes(B, H, S)), window=W)
    _sync()
    oout, olse = oracle.attn_fwd(qkv, B, H, S, window=W)
    assert_same_bits(host(out, np.uint16), oout, "out")
    assert_same_bits(host(d, np.uint16), oracle.attn_bwd(dout, qkv, oout, olse, B, H, S, window=W), "gradients")


def _scores(q, k, v, g, out, lse):
    """P and dS of one head for every pair, as bf16, in the arithmetic of the primitives; all arguments binary32."""
    op, scale, S = oracle.prim, np.full((len(q), len(q)), 0.08838834764831845, F), len(q)
    s, dp = np.zeros((S, S), F), np.zeros((S, S), F)
    for c in range(128):
        s = op("add", s, op("mul", np.broadcast_to(q[:, c, None], (S, S)), np.broadcast_to(k[None, :, c], (S, S))))
        dp = op("add", dp, op("mul", np.broadcast_to(g[:, c, None], (S, S)), np.broadcast_to(v[None, :, c], (S, S))))
    t = op("mul", g, out)
    while t.shape[1] > 1:
        t = op("add", t[:, 0::2], t[:, 1::2])
    p = op("exp", op("sub", op("mul", s, scale), np.broadcast_to(lse[:, None], (S, S))))
    return synth.to_bf16(p), synth.to_bf16(op("mul", op("mul", p, op("sub", dp, np.broadcast_to(t, (S, S)))), scale))


# the three forms of the kernel that forms P and dS (few blocks; up to seven quarters of the SMs; epilogue warps) on the inputs that their branches are
# for: a logsumexp that is not the row's own (positive arguments of the exponential), weights that vanish, non-finite values, and products of
# dO and v that underflow, all of them in one slab of 16 dimensions, in which v alone is below 2^-63 (heads take turns through the eight).
# P and dS themselves, of the pairs that are visible, from the workspace: nine heads
@pytest.mark.parametrize("form", ["few", "lone", "tall"])
@pytest.mark.parametrize("per_head,S,W", [(3, 256, 0), (5, 320, 128)])
@pytest.mark.parametrize("kind", ["logsumexp", "saturated", "non-finite", "underflow"])
def test_attention_backward_scores(det, form, per_head, S, W, kind):
    B, H = 1, 8 if form == "few" else 7 * det.det_device_sm_count() // 4 // per_head + (form == "tall")
    HD = H * 128
    rng = np.random.default_rng(S + H)
    x = synth.from_bf16(synth.normal_bf16((S, 3 * HD), 1.0, seed=H, tid=1)).reshape(S, 3, H, 128).copy()
    g = synth.from_bf16(synth.normal_bf16((S, HD), 0.1, seed=H, tid=2)).reshape(S, H, 128).copy()
    if kind == "saturated":
        x[:, 0] *= F(40.0)
    elif kind == "non-finite":                                     # in three heads of every eight, at both ends of the sequence and inside
        x[S - 1, 0, 1::8, 5], x[3, 1, 4::8, 70], x[130, 2, 6::8, 127] = np.nan, np.inf, -np.inf
    elif kind == "underflow":
        x[:, 2], g[:] = 0, 0
        for h in range(H):
            d = 16 * (h % 8)
            x[:, 2, h, d:d + 16] = F(2.0 ** -65) * (1 + rng.integers(0, 4, (S, 16)) / 8)
            x[:, 2, h, d] = rng.choice(np.array([-1, 1], F), S) * F(2.0 ** -56)
            g[:, h, d:d + 16] = F(2.0 ** -62) * (1 + rng.integers(0, 4, (S, 16)) / 8)
            g[:, h, d] = F(2.0 ** -60)
    qkv, dout = synth.to_bf16(x.reshape(S, 3 * HD)), synth.to_bf16(g.reshape(S, HD))
    x, g = synth.from_bf16(qkv).reshape(S, 3, H, 128), synth.from_bf16(dout).reshape(S, H, 128)
    out, lse = oracle.attn_fwd(qkv, B, H, S, window=W)
    if kind == "logsumexp":
        lse -= rng.choice(np.array([0.0, 0.75, 3.0, -2.0], F), lse.shape)
    d_in, d, scratch = dev(qkv), empty((S, 3 * HD), np.uint16), ws(det.det_attn_bwd_ws_bytes(B, H, S))
    q, o = d_in.data_ptr(), d.data_ptr()
    det.det_attn_bwd(dev(dout), q, q + 2 * HD, q + 4 * HD, dev(out), dev(lse), 3 * HD, HD, B, H, S, o, o + 2 * HD, o + 4 * HD, 3 * HD, scratch, window=W)
    _sync()
    raw, n = host(scratch), H * S * S * 2
    got = [raw[at:at + n].view(np.uint16).reshape(H, S, S) for at in (0, -(-n // 256) * 256)]
    i, j = np.indices((S, S))
    vis = (j <= i) & ((W == 0) | (j > i - W))
    o = synth.from_bf16(out).reshape(S, H, 128)
    for h in [8 * (r * (H // 8) // 8) + r for r in range(8)] + [H - 1]:
        for name, a, b in zip(("P", "dS"), got, _scores(x[:, 0, h], x[:, 1, h], x[:, 2, h], g[:, h], o[:, h], lse[0, h])):
            a, b = a[h][vis], b[vis]
            nan = np.isnan(synth.from_bf16(b))
            assert np.array_equal(np.isnan(synth.from_bf16(a)), nan) and (kind == "non-finite" or not nan.any())
            assert_same_bits(a[~nan], b[~nan], "%s of head %d" % (name, h))
            assert kind == "non-finite" or np.count_nonzero(synth.from_bf16(b)) > S


# the backward's blocks in equal runs, in runs with short ones at the end, and by whole query blocks: heads of one call against the
# same heads in calls of their own
@pytest.mark.parametrize("B,H,S", [(1, 3, 1344), (1, 18, 2048), (4, 16, 2048)])
def test_attention_backward_heads_apart(det, B, H, S):
    def run(B, H, qkv, dout):
        HD, x = H * 128, dev(qkv)
        q = x.data_ptr()
        out, lse, dqkv = empty((B * S, HD), np.uint16), empty((B, H, S), F), empty((B * S, 3 * HD), np.uint16)
        det.det_attn_fwd(q, q + 2 * HD, q + 4 * HD, 3 * HD, B, H, S, out, HD, lse)
        d = dqkv.data_ptr()
        det.det_attn_bwd(dev(dout), q, q + 2 * HD, q + 4 * HD, out, lse, 3 * HD, HD, B, H, S, d, d + 2 * HD, d + 4 * HD, 3 * HD,
                         ws(det.det_attn_bwd_ws_bytes(B, H, S)))
        _sync()
        return host(dqkv, np.uint16).reshape(B, S, 3, H, 128)
    qkv = synth.normal_bf16((B * S, 3 * H * 128), 1.0, seed=H, tid=1).reshape(B, S, 3, H, 128)
    dout = synth.normal_bf16((B * S, H * 128), 0.1, seed=H, tid=2).reshape(B, S, H, 128)
    got = run(B, H, qkv, dout)
    for b, h in ((0, 0), (B - 1, H // 2), (B - 1, H - 1)):
        want = run(1, 1, np.ascontiguousarray(qkv[b:b + 1, :, :, h:h + 1]), np.ascontiguousarray(dout[b:b + 1, :, h:h + 1]))
        assert_same_bits(got[b, :, :, h], want[0, :, :, 0], "gradients of head %d" % h)


# the two-lane exponential: a dense grid of arguments, the ends of the kept range, subnormal, infinite and NaN arguments
def test_two_lane_exponential(det):
    x = np.concatenate([np.linspace(-90, 0, 400001), np.linspace(-87.4, -87.2, 20001), [0.0, -0.0, -1e-40, -1e-30, -200.0, -1e30, -np.inf, np.nan]]).astype(F)
    a, got, want = dev(x), empty(x.shape, F), empty(x.shape, F)
    det.det_test_prim(11, a, None, got)
    det.det_test_prim(5, a, None, want)
    _sync()
    n = np.isnan(x)
    assert_same_bits(host(got)[~n], host(want)[~n], "exp")
    assert np.isnan(host(got)[n]).all()


# global norm over many tensors in common launches: more tensors than one launch takes, empty and one-element ones, lengths
# around a chunk of 16384 and around the second level (16384 chunks would be 2^28 elements: 40 chunks stand for it)
@pytest.mark.parametrize("sizes", [[0], [1], [16384, 16385, 0, 1, 300, 16383, 655361, 8, 65536], [(977 * i) % 40000 for i in range(520)]])
def test_grad_norm_many_tensors(det, sizes):
    import torch
    g = [synth.normal_f32((n,), 1e-3, seed=len(sizes), tid=i) if n else np.zeros(0, F) for i, n in enumerate(sizes)]
    if sizes == [1]:
        g = [np.array([1e-40], F)]              # a lone subnormal is flushed
    d = [dev(x) for x in g]
    norm, coef, status = empty((1,), F), empty((1,), F), torch.zeros(1, dtype=torch.int32, device="cuda")
    det.det_grad_norm(d, 0.5, norm, coef, ws(det.det_grad_norm_ws_bytes(d)), status)
    _sync()
    n_o, c_o = oracle.grad_norm(g, 0.5)
    assert_same_bits(host(norm), np.array([n_o], F), "norm")
    assert_same_bits(host(coef), np.array([c_o], F), "coef")
    assert int(status.item()) == 0


# AdamW of many tensors in one launch with the clip coefficient applied on the way: both parameter types, lengths off the
# 4- and 1024-element grid, empty tensors, more tensors than one launch takes, different decay per tensor
@pytest.mark.parametrize("sizes,clip", [([1, 3, 4, 5, 1023, 1024, 1025, 0, 4100], True), ([2048, 7], False), ([(37 * i) % 600 for i in range(300)], True)])
def test_adamw_many_tensors(det, sizes, clip):
    rng = np.random.default_rng(len(sizes))
    coef = F(0.3125 + 1e-3)
    kinds = [int(i % 3 != 2) for i in range(len(sizes))]
    wd = [0.1 if i % 2 else 0.0 for i in range(len(sizes))]
    p = [synth.to_bf16(rng.standard_normal(n, dtype=F)) if k else rng.standard_normal(n, dtype=F) for n, k in zip(sizes, kinds)]
    g, m = [[rng.standard_normal(n, dtype=F) * F(s) for n in sizes] for s in (1e-2, 1e-3)]
    v = [np.abs(rng.standard_normal(n, dtype=F)) * F(1e-5) for n in sizes]
    dp, dg, dm, dv = [[dev(x) for x in t] for t in (p, g, m, v)]
    descs = [det.det_adamw_desc(3e-4, 0.9, 0.95, 1e-8, w, 3) for w in wd]
    det.det_adamw_batch(descs, kinds, dp, dg, dm, dv, dev(np.array([coef], F)) if clip else None)
    _sync()
    for i, n in enumerate(sizes):
        if not n:
            continue
        go = oracle.scale(g[i], coef) if clip else g[i]
        po, mo, vo = oracle.adamw(p[i], go, m[i], v[i], 3e-4, 0.9, 0.95, 1e-8, wd[i], 3)
        assert_same_bits(host(dg[i]), go, "g %d" % i)
        assert_same_bits(host(dp[i], p[i].dtype), po, "p %d" % i)
        assert_same_bits(host(dm[i]), mo, "m %d" % i)
        assert_same_bits(host(dv[i]), vo, "v %d" % i)


# the rotated transposed weight codes: codes at both ends of the range (all of one sign, so that the plain
# sum is +-2^14), a column block without a partner, more than one tile per CTA
@pytest.mark.parametrize("N,K", [(128, 128), (256, 384), (3072, 8320)])
def test_weight_rotation(det, N, K):
    rng = np.random.default_rng(N + K)
    W = np.where(rng.random((N, K)) < 0.5, -1.0, 1.0)
    W[:, 0], W[:, 1], W[:128, K - 1] = 1.0, -1.0, -1.0
    W[:, 2:64:3] = 1e-3 * rng.integers(-128, 128, (N, len(range(2, 64, 3))))
    q = np.clip(np.rint(synth.from_bf16(synth.to_bf16(W.astype(F))) * (F(1.0) / F(1e-3))), -128, 127).astype(np.int64)
    v = q.reshape(N // 128, 128, K)
    for h in (1, 2, 4, 8, 16, 32, 64):
        v = v.reshape(N // 128, 64 // h, 2, h, K)
        v = np.stack((v[:, :, 0] + v[:, :, 1], v[:, :, 0] - v[:, :, 1]), axis=2).reshape(N // 128, 128, K)
    am = np.abs(v).max()
    want = np.rint(v.astype(F) * (F(127.0) / F(am))).astype(np.int8).reshape(N, K).T
    qW, qWt, s_u = empty((N, K), np.int8), empty((K, N), np.int8), empty((1,), F)
    det.det_lsq_quantize_weight(dev(synth.to_bf16(W.astype(F))), dev(np.full(N, 1e-3, F)), N, K, 128, qW, qWt, s_u, ws(256))
    _sync()
    assert_same_bits(host(qW, np.int8), q.astype(np.int8), "codes")
    assert_same_bits(host(qWt, np.int8), np.ascontiguousarray(want), "rotated codes")
    assert_same_bits(host(s_u), np.array([F(am) / F(127.0)], F), "step")


# LSQ linear at sizes where the tile of the int8 GEMMs changes (64, 128, 256 columns, CTA pairs), with a last round that is
# nearly empty and with dimensions that only narrow tiles divide; the operand preparation one item per CTA, two, and (the last) more tiles of dY and of Z than CTAs,
# so that a CTA's buffers change places
@pytest.mark.parametrize("M,N,K", [(128, 128, 128), (384, 640, 384), (1024, 3072, 1024), (1664, 3072, 1024), (2048, 3072, 1024), (10240, 768, 896)])
def test_linear_tiles(det, M, N, K):
    import torch
    X, W = synth.normal_bf16((M, K), 1.0, seed=M, tid=1), synth.normal_bf16((N, K), 0.02, seed=M, tid=2)
    dY = synth.normal_bf16((M, N), 0.01, seed=M, tid=3)
    X[::7, ::11] = synth.to_bf16(np.array([40.0], F))[0]           # outside the quantiser's range: masked gradient, clamped phi
    sw, sx = oracle.lsq_weight_scale(W), oracle.lsq_act_scale_init(synth.normal_bf16((M, K), 1.0, seed=M, tid=1))
    oY, oqX, oqW = oracle.linear_fwd(X, W, sx, sw)
    odX, odW, ods = oracle.linear_bwd(dY, X, W, sx, sw, hb=128)
    dX_, dW_, s_w, s_x = dev(X), dev(W), dev(sw), dev(sx)
    qW, qWt, s_u = empty((N, K), np.int8), empty((K, N), np.int8), empty((1,), F)
    det.det_lsq_quantize_weight(dW_, s_w, N, K, 128, qW, qWt, s_u, ws(det.det_lsq_quantize_weight_ws_bytes(N, K)))
    Y, qX, status = empty((M, N), np.uint16), empty((M, K), np.int8), torch.zeros(1, dtype=torch.int32, device="cuda")
    det.det_linear_fwd(dX_, qW, s_x, s_w, M, N, K, Y, qX, status)
    gX, gW, gs = empty((M, K), np.uint16), empty((N, K), F), empty((1,), F)
    det.det_linear_bwd(dev(dY), dX_, qX, dW_, qWt, s_x, s_w, s_u, M, N, K, 128, gX, gW, gs, ws(det.det_linear_bwd_ws_bytes(M, N, K)), status)
    _sync()
    assert int(status.item()) == 0
    assert_same_bits(host(Y, np.uint16), oY, "Y")
    assert_same_bits(host(gX, np.uint16), odX, "dX")
    assert_same_bits(host(gW), odW, "dW")
    assert_same_bits(host(gs), ods, "ds_x")


# the two gradient products of a linear in one launch: one tile each, either product first, CTAs with and without a tile of the first one, widths
# that only 64 columns divide, with and without the rotation; and in two launches on either side of the rule
@pytest.mark.parametrize("M,N,K,hb", [(128, 128, 128, 128), (2048, 128, 128, 0), (1280, 1408, 384, 128), (640, 384, 896, 0), (1536, 1408, 640, 128),
                                      (1920, 896, 256, 128), (512, 2944, 256, 128), (3968, 128, 256, 0)])
def test_linear_gradients_together(det, M, N, K, hb):
    import torch
    X, W = synth.normal_bf16((M, K), 1.0, seed=N, tid=1), synth.normal_bf16((N, K), 0.02, seed=N, tid=2)
    dY = synth.normal_bf16((M, N), 0.01, seed=N, tid=3)
    sw, sx = oracle.lsq_weight_scale(W), oracle.lsq_act_scale_init(X)
    odX, odW, ods = oracle.linear_bwd(dY, X, W, sx, sw, hb=hb)
    dX_, dW_, s_w, s_x = dev(X), dev(W), dev(sw), dev(sx)
    qW, qWt, s_u = empty((N, K), np.int8), empty((K, N), np.int8), empty((1,), F)
    det.det_lsq_quantize_weight(dW_, s_w, N, K, hb, qW, qWt, s_u, ws(det.det_lsq_quantize_weight_ws_bytes(N, K)))
    Y, qX, status = empty((M, N), np.uint16), empty((M, K), np.int8), torch.zeros(1, dtype=torch.int32, device="cuda")
    det.det_linear_fwd(dX_, qW, s_x, s_w, M, N, K, Y, qX, status)
    gX, gW, gs = empty((M, K), np.uint16), empty((N, K), F), empty((1,), F)
    det.det_linear_bwd(dev(dY), dX_, qX, dW_, qWt, s_x, s_w, s_u, M, N, K, hb, gX, gW, gs, ws(det.det_linear_bwd_ws_bytes(M, N, K)), status)
    _sync()
    assert int(status.item()) == 0
    assert_same_bits(host(gX, np.uint16), odX, "dX")
    assert_same_bits(host(gW), odW, "dW")
    assert_same_bits(host(gs), ods, "ds_x")


# the same in one launch with more tiles than SMs, so that a CTA passes from a tile of one product to one of the other: each product first, all three
# widths, CTAs that take two and three tiles of the second product while others are at the first, first products of one and of two tiles a CTA.
# prep: launches of the operand preparation, without the rotation and with it (two passes for few tiles, two times two for many)
@pytest.mark.parametrize("M,N,K,hb,prep", [(128, 128, 4992, 128, 2), (4224, 1920, 256, 0, 5), (7296, 2304, 256, 0, 5), (128, 3840, 640, 128, 2),
                                           (6528, 128, 768, 0, 5), (128, 4224, 1280, 0, 5), (6144, 128, 1024, 0, 5), (512, 3072, 1792, 0, 5)])
def test_linear_gradients_together_many_tiles(det, M, N, K, hb, prep):
    import torch
    X, W = synth.normal_bf16((M, K), 1.0, seed=N, tid=1), synth.normal_bf16((N, K), 0.02, seed=N, tid=2)
    dY = synth.normal_bf16((M, N), 0.01, seed=N, tid=3)
    sw, sx = oracle.lsq_weight_scale(W), oracle.lsq_act_scale_init(X)
    odX, odW, ods = oracle.linear_bwd(dY, X, W, sx, sw, hb=hb)
    dX_, dW_, s_w, s_x = dev(X), dev(W), dev(sw), dev(sx)
    qW, qWt, s_u = empty((N, K), np.int8), empty((K, N), np.int8), empty((1,), F)
    det.det_lsq_quantize_weight(dW_, s_w, N, K, hb, qW, qWt, s_u, ws(det.det_lsq_quantize_weight_ws_bytes(N, K)))
    Y, qX, status = empty((M, N), np.uint16), empty((M, K), np.int8), torch.zeros(1, dtype=torch.int32, device="cuda")
    det.det_linear_fwd(dX_, qW, s_x, s_w, M, N, K, Y, qX, status)
    gX, gW, gs = empty((M, K), np.uint16), empty((N, K), F), empty((1,), F)
    before = det.det_launch_count()
    det.det_linear_bwd(dev(dY), dX_, qX, dW_, qWt, s_x, s_w, s_u, M, N, K, hb, gX, gW, gs, ws(det.det_linear_bwd_ws_bytes(M, N, K)), status)
    assert det.det_launch_count() - before == prep + 1 + (1 if M * K // 64 <= 16384 else 2)      # the products in one, the sum of the step gradient
    _sync()
    assert int(status.item()) == 0
    assert_same_bits(host(gX, np.uint16), odX, "dX")
    assert_same_bits(host(gW), odW, "dW")
    assert_same_bits(host(gs), ods, "ds_x")


# the norms with the residual stream beside them: rows off the block of eight, D off the leaf of 256, with and without codes
@pytest.mark.parametrize("rows,D,q", [(1, 8, True), (13, 1000, False), (300, 2048, True), (64, 384, True), (21, 256, True), (22, 512, False),
                                      (23, 1024, True), (9, 1032, True), (515, 200, False)])
def test_norms_with_residual(det, rows, D, q):
    a, b, dy, res = [synth.normal_bf16((rows, D), 1.0, seed=rows, tid=t) for t in range(4)]
    gain = synth.normal_bf16((D,), 0.1, mean=1.0, seed=rows, tid=9)
    s = np.array([0.03], F)
    h, y, rstd, qy = empty((rows, D), np.uint16), empty((rows, D), np.uint16), empty((rows,), F), empty((rows, D), np.int8)
    det.det_residual_rmsnorm_fwd(dev(a), dev(b), dev(gain), rows, D, 1e-6, h, y, rstd, dev(s) if q else None, qy if q else None)
    _sync()
    ho = oracle.residual_add(a, b)
    yo, ro = oracle.rmsnorm_fwd(ho, gain, 1e-6, bf=True)
    assert_same_bits(host(h, np.uint16), ho, "sum")
    assert_same_bits(host(y, np.uint16), yo, "y")
    assert_same_bits(host(rstd), ro.reshape(-1), "rstd")
    if q:
        assert_same_bits(host(qy).reshape(-1), np.asarray(oracle.lsq_quantize(yo, s, False)).reshape(-1).view(np.int8), "codes")
    dx, dg = dev(res), empty((D,), F)
    det.det_rmsnorm_bwd_residual(dev(dy), dev(ho), dev(gain), rstd, rows, D, dx, dx, dg, ws(det.det_rmsnorm_bwd_ws_bytes(rows, D)))
    _sync()
    dxo, dgo = oracle.rmsnorm_bwd(dy, ho, gain, ro, bf=True)
    assert_same_bits(host(dx, np.uint16), oracle.residual_add(res, dxo), "dx")
    assert_same_bits(host(dg), dgo.reshape(-1), "dgain")


# a weight of many tiles stays on the caller's stream: it does not wait for another stream's linear backward, whose kernels on the
# auxiliary streams stand behind 0.2 s of other work
def test_weight_quantisation_waits_for_nobody(det):
    import time
    import torch
    M, N, K = 2048, 3072, 1024                                     # large enough for the auxiliary streams
    X, dY, W = [dev(synth.normal_bf16(s, 0.1, seed=1, tid=t)) for t, s in enumerate(((M, K), (M, N), (N, K)))]
    sw, one = dev(np.full(N, 1e-3, F)), dev(np.ones(1, F))
    qX, qWt, status = dev(np.ones((M, K), np.int8)), dev(np.ones((K, N), np.int8)), torch.zeros(1, dtype=torch.int32, device="cuda")
    dX, dW, ds, wb = empty((M, K), np.uint16), empty((N, K), F), empty((1,), F), ws(det.det_linear_bwd_ws_bytes(M, N, K))
    big = dev(synth.normal_bf16((3072, 8320), 0.1, seed=2, tid=0))
    out = [(empty((3072, 8320), np.int8), empty((8320, 3072), np.int8), empty((1,), F), ws(256)) for _ in range(8)]
    backward = lambda: det.det_linear_bwd(dY, X, qX, W, qWt, one, sw, one, M, N, K, 128, dX, dW, ds, wb, status)
    weights = lambda o: det.det_lsq_quantize_weight(big, sw, 3072, 8320, 128, o[0], o[1], o[2], o[3])
    backward()                                                     # everything is loaded before it counts
    weights(out[0])
    _sync()
    first, others, slept = torch.cuda.Stream(), [torch.cuda.Stream() for _ in out], torch.cuda.Event()
    with torch.cuda.stream(first):
        torch.cuda._sleep(400_000_000)
        slept.record()
        backward()
    done = []
    for s, o in zip(others, out):                                  # several: two streams can share a hardware queue
        with torch.cuda.stream(s):
            weights(o)
            done.append(torch.cuda.Event())
            done[-1].record()
    free = False
    end = time.monotonic() + 30
    while not free and not slept.query() and time.monotonic() < end:
        free = any(e.query() for e in done) and not slept.query()
    _sync()
    assert free


# the forward pass with int8 P.V over many key blocks: nine and eleven per row block (with the last row block ragged), six in a window,
# so that the two value buffers, the four block scales and the barriers' parities come round again; every block of 128 keys has a value
# range of its own, so that a stale scale or buffer shows
@pytest.mark.parametrize("B,H,Hkv,S,W", [(1, 2, 2, 1088, 0), (2, 2, 1, 1344, 0), (1, 4, 2, 1472, 640)])
def test_int8_pv_many_blocks(det, B, H, Hkv, S, W):
    import torch
    HD, KD = H * 128, Hkv * 128
    ld = HD + 2 * KD
    x = synth.from_bf16(synth.normal_bf16((B * S, ld), 1.0, seed=S, tid=1)).astype(F)
    x[:, HD + KD:] *= (F(3.0) ** ((np.arange(B * S) % S // 128 * 5) % 7 - 3).astype(F))[:, None]
    qkv = synth.to_bf16(x)
    d = dev(qkv)
    q = d.data_ptr()
    out, lse, status = empty((B * S, HD), np.uint16), empty((B, H, S), F), torch.zeros(1, dtype=torch.int32, device="cuda")
    det.det_attn_fwd_int8pv(q, q + 2 * HD, q + 2 * (HD + KD), ld, B, H, S, out, HD, lse, status, Hkv=Hkv, window=W)
    _sync()
    assert int(status.item()) == 0
    oout, olse = oracle.attn_fwd(qkv, B, H, S, Hkv=Hkv, window=W, int8_pv=True)
    assert_same_bits(host(lse), olse, "lse")
    assert_same_bits(host(out, np.uint16), oout, "out")
