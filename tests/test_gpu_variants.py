"""GPU parity of kernel variants that a rule on sizes chooses, at the sizes where each can go wrong: edges of
its tiles, remainders, the smallest and the largest shapes of its range."""
import numpy as np
import pytest
import torch

from oracle import ap_oracle as orc
from paper_2012_02030_b200 import inputs
from tests import parity_util as pu
from tests import test_gpu_parity as tp

pytestmark = pytest.mark.gpu

W = inputs.WORKLOADS


@pytest.fixture(scope="module")
def ap():
    from paper_2012_02030_b200 import binding

    assert torch.cuda.is_available()
    return binding


@pytest.mark.parametrize("d", [64, 128])
@pytest.mark.parametrize("shape", [(1, 1, 9, 130), (5, 4, 250, 70), (10, 4, 250, 140)])  # 8, 16, 32 rows per block
def test_fp32_forward_rows_per_block(ap, shape, d):
    B, H, Lq, Lk = shape
    w = W["tiny"].scaled(B=B, H=H, Lq=Lq, Lk=Lk, d=d, dtype="f32")
    mask = inputs.random_mask(H, Lq, Lk, 0.2, seed=501, empty_rows=(3,))
    q, k, v = inputs.eval_qkv(w)
    tiles = ap.Tiles(H, Lq, Lk)
    ap.ap_mask_to_tiles(mask.cuda(), tiles)
    out = ap.ap_sparse_attention_fwd(q.cuda(), k.cuda(), v.cuda(), tiles, torch.full_like(q, float("nan"), device="cuda"))
    assert ap.ap_device_status() == ap.AP_OK
    ref = orc.attention_fwd(inputs.widen(q), inputs.widen(k), inputs.widen(v), mask.numpy())
    pu.assert_close_attention(out, ref, "f32", str(shape))
    assert np.all(out[:, :, 3].cpu().numpy() == 0.0)


@pytest.mark.parametrize("dtype,d", [("bf16", 64), ("f16", 64), ("bf16", 128)])
@pytest.mark.parametrize("columns", [13, 40])
def test_forward_rounds_that_one_softmax_group_sits_out(ap, dtype, d, columns):
    """Many short lists in a row: every round has one slot (or three), so that one of the softmax groups has no chunk of
    any round (or only a partial one) and nothing to slow it down but the barriers."""
    B, H, L = 16, 5, 2048
    w = W["tiny"].scaled(B=B, H=H, Lq=L, Lk=L, d=d, dtype=dtype)
    mask = torch.zeros((H, L, L), dtype=torch.uint8)
    mask[:, :, :columns] = inputs.random_mask(H, L, columns, 0.5, seed=502)
    mask[:, 7] = 0
    q, k, v = inputs.eval_qkv(w)
    v = v * 0.5  # outputs near single values of V stay below 4, where half an ulp of bf16 is 2^-7 < 1e-2
    tiles = ap.Tiles(H, L, L)
    ap.ap_mask_to_tiles(mask.cuda(), tiles)
    out = ap.ap_sparse_attention_fwd(q.cuda(), k.cuda(), v.cuda(), tiles, torch.full_like(q, float("nan"), device="cuda"))
    assert ap.ap_device_status() == ap.AP_OK
    n = columns  # the keys beyond are kept nowhere
    ref = orc.attention_fwd(inputs.widen(q), inputs.widen(k[:, :, :n].contiguous()), inputs.widen(v[:, :, :n].contiguous()),
                            mask[:, :, :n].contiguous().numpy())
    assert np.abs(ref).max() < 4.0
    pu.assert_close_attention(out, ref, dtype, str(columns))
    assert np.all(out[:, :, 7].float().cpu().numpy() == 0.0)


def _scores(H, Lq, Lk, seed):
    """One head each of distinct, quantised (ties by the thousand), skewed and, last, constant values."""
    acc = np.random.default_rng(seed).random((H, Lq, Lk), dtype=np.float32)
    acc[1] = np.round(acc[1] * 32) / 32
    acc[2] = acc[2] ** 8
    acc[-1] = 0.75
    return acc


@pytest.mark.parametrize("layer", [False, True])
@pytest.mark.parametrize("H,Lq,Lk,causal", [(4, 1792, 1792, False),    # rows on 32-byte boundaries
                                            (8, 1801, 1804, True),     # rows on 16-byte boundaries, four memory keys
                                            (4, 1800, 1801, False)])   # rows anywhere
def test_build_mask_from_drawn_pivots(ap, H, Lq, Lk, causal, layer):
    """More than 12 * 2^20 entries in all: pivots from drawn entries, one pass between them, the select over the collected
    entries; the constant head overflows its buffer and is selected over the accumulator."""
    acc = _scores(H, Lq, Lk, 503)
    w = W["tiny"].scaled(H=H, Lq=Lq, Lk=Lk, causal=causal, keep_diag=causal, keep_frac=0.07)
    mask, tiles, nnz = pu.gpu_build_mask(ap, torch.from_numpy(acc).cuda(), w, layer=layer)
    want, want_nnz = (orc.build_mask_layer if layer else orc.build_mask)(acc, 0.07, causal, causal)
    np.testing.assert_array_equal(mask.cpu().numpy(), want)
    np.testing.assert_array_equal(nnz.cpu().numpy(), want_nnz)
    pu.assert_tiles_equal(tiles.to_host(), orc.mask_to_tiles(want))


def test_build_mask_scores_16_bytes_past_a_sector(ap):
    H, L = 3, 256
    acc = _scores(H, L, L, 504)
    want, _ = orc.build_mask(acc, 0.2, True, True)
    acc_dev = torch.zeros(H * L * L + 4, device="cuda")[4:].view(H, L, L).copy_(torch.from_numpy(acc))
    mask = torch.full((H, L, L), 7, dtype=torch.uint8, device="cuda")
    ap.ap_build_mask(acc_dev, 0.2, True, True, mask=mask)
    assert ap.ap_device_status() == ap.AP_OK
    np.testing.assert_array_equal(mask.cpu().numpy(), want)


@pytest.mark.parametrize("B,H,Lq,Lk,causal", [(7, 2, 512, 512, True),    # chunks of samples, an odd number of them
                                              (5, 1, 260, 388, True),    # memory keys, ragged
                                              (16, 3, 130, 64, False),   # one key tile, a query tile of two rows
                                              (3, 1, 70, 301, False),    # rows that no tensor map can describe, ...
                                              (18, 2, 200, 387, True)])  # ... in chunks
def test_accumulate_chunks_of_samples(ap, B, H, Lq, Lk, causal):
    """Fewer units of work than SMs: each query tile's samples are cut into chunks of about equal numbers of visits."""
    w = W["tiny"].scaled(B=B, H=H, Lq=Lq, Lk=Lk, d=64, dtype="bf16", causal=causal)
    bias = inputs.calib_bias(w)
    acc = pu.gpu_accumulate(ap, w, 2, bias.cuda())
    assert ap.ap_device_status() == ap.AP_OK
    assert torch.equal(acc, pu.gpu_accumulate(ap, w, 2, bias.cuda()))
    want = pu.oracle_accumulate(w, 2, bias)
    tol = tp._acc_tolerance(w.dtype)
    np.testing.assert_allclose(acc.cpu().numpy(), want, rtol=tol["rtol"], atol=tol["atol"] * 2 * B)


@pytest.mark.parametrize("dtype,d", [("bf16", 64), ("f16", 64), ("bf16", 128)])
def test_forward_three_query_tiles(ap, dtype, d):
    """A pair and a lone query tile per head, over more units than SMs: the grid has no factor in common with a head's units."""
    B, H, Lq, Lk = 16, 8, 300, 333
    w = W["tiny"].scaled(B=B, H=H, Lq=Lq, Lk=Lk, d=d, dtype=dtype)
    mask = inputs.random_mask(H, Lq, Lk, 0.2, seed=505, empty_rows=(299,))
    q, k, v = inputs.eval_qkv(w)
    v = v * 0.5  # |O| below 4, see above
    tiles = ap.Tiles(H, Lq, Lk)
    ap.ap_mask_to_tiles(mask.cuda(), tiles)
    # an output that starts 16 bytes past a 32-byte boundary is written in 16-byte pieces
    plain = torch.full_like(q, float("nan"), device="cuda")
    odd = torch.full((q.numel() + 8,), float("nan"), dtype=q.dtype, device="cuda")[8:].view(q.shape)
    for out in (plain, odd):
        ap.ap_sparse_attention_fwd(q.cuda(), k.cuda(), v.cuda(), tiles, out)
    assert ap.ap_device_status() == ap.AP_OK
    assert torch.equal(plain, odd)
    ref = orc.attention_fwd(inputs.widen(q), inputs.widen(k), inputs.widen(v), mask.numpy())
    assert np.abs(ref).max() < 4.0
    pu.assert_close_attention(plain, ref, dtype)


@pytest.mark.parametrize("dtype,d,tol", [("bf16", 64, 1e-2), ("bf16", 128, 1e-2), ("f16", 64, 2e-3), ("f16", 128, 2e-3)])
@pytest.mark.parametrize("Lq,Lk", [(1024, 1024), (1030, 901)])
def test_backward_gathered_key_blocks(ap, dtype, d, tol, Lq, Lk):
    """Heavy key groups (sinks, strided columns, the last, partial group) among a band: they come last in the key order and
    blocks gather them from several tiles.  The second head keeps the band alone and a key tile that nobody keeps."""
    w = W["tiny"].scaled(B=1, H=2, Lq=Lq, Lk=Lk, d=d, dtype=dtype)
    i, j = torch.arange(Lq)[:, None], torch.arange(Lk)[None, :]
    band = (i * Lk // Lq - j).abs() <= 20
    mask = torch.stack([band | (j < 3) | (j % 200 == 150) | (j == Lk - 1), band & (j // 128 != 2)]).to(torch.uint8)
    tp._bwd_case(ap, w, mask, tol)


@pytest.mark.parametrize("dtype", ["bf16", "f16"])
@pytest.mark.parametrize("spread", [0.0, 1e-3, 1.0])
def test_entmax_forward_candidate_lists(ap, dtype, spread):
    """More kept entries per row than a candidate list holds: equal scores (every entry is a candidate, no list can be
    pruned), scores within 1e-3 of one another (the same), and spread-out ones (pruned once or more)."""
    w = W["tiny"].scaled(B=1, H=2, Lq=200, Lk=520, d=64, dtype=dtype)
    mask = inputs.random_mask(w.H, w.Lq, w.Lk, 0.9, seed=506, empty_rows=(9,))
    mask[1, :, 60:] = 0                            # the second head: lists that just fit or just do not
    tp._entmax_fwd_case(ap, w, mask, scale=spread / 8 if spread else 1e-30)


@pytest.mark.parametrize("Lk", [33, 260])
def test_fp32_accumulate_key_rows_16_bytes_past_a_sector(ap, Lk):
    """Key rows that start on 32-byte boundaries are read with wider loads: the same numbers either way."""
    w = W["tiny"].scaled(B=3, H=2, Lq=29, Lk=Lk, d=64, dtype="f32", causal=False)
    q, k = (t.cuda() for t in inputs.calib_qk(w, 0))
    odd = torch.zeros(k.numel() + 4, device="cuda")[4:].view(k.shape).copy_(k)
    got = [torch.zeros((w.H, w.Lq, w.Lk), device="cuda") for _ in range(2)]
    for acc, keys in zip(got, (k, odd)):
        ap.ap_accumulate_attention(acc, q, keys, None, causal=False)
    assert ap.ap_device_status() == ap.AP_OK
    assert torch.equal(*got)
    want = np.zeros((w.H, w.Lq, w.Lk))
    orc.accumulate(want, inputs.widen(q.cpu()), inputs.widen(k.cpu()), None, causal=False)
    tol = tp._acc_tolerance("f32")
    np.testing.assert_allclose(got[0].cpu().numpy(), want, rtol=tol["rtol"], atol=tol["atol"] * w.B)


@pytest.mark.parametrize("d", [64, 128])
def test_fp16_backward_many_items_of_few_rounds(ap, d):
    """fp16 tensors sweep an item's rounds twice, the first time without a dQ: many items of one round each beside items of
    several, so that a first sweep runs ahead of what reads out the item before."""
    B, H, L = 24, 4, 640
    w = W["tiny"].scaled(B=B, H=H, Lq=L, Lk=L, d=d, dtype="f16")
    i, j = torch.arange(L)[:, None], torch.arange(L)[None, :]
    few = (j < 4) | (i == j)                           # one or two rounds
    many = (j % 8 == i % 8) & (i // 128 % 2 == 1) | few  # every other query tile: five rounds
    mask = torch.stack([few, many, few, many]).to(torch.uint8)
    q, k, v = (t.cuda() for t in inputs.eval_qkv(w))
    d_o = torch.randn(q.shape, generator=torch.Generator(device="cuda").manual_seed(507), device="cuda").to(q.dtype)
    tiles = ap.Tiles(H, L, L)
    ap.ap_mask_to_tiles(mask.cuda(), tiles)
    out = ap.ap_sparse_attention_fwd(q, k, v, tiles)
    for _ in range(20):
        got = ap.ap_sparse_attention_bwd(q, k, v, out, d_o, tiles)
    assert ap.ap_device_status() == ap.AP_OK
    for b in (0, B - 1):
        want = orc.attention_bwd(*(inputs.widen(t[b:b + 1].cpu()) for t in (q, k, v, d_o)), mask.numpy())
        for x, ref in zip(got, want):
            assert np.linalg.norm(x[b].float().cpu().numpy() - ref[0]) <= 2e-3 * np.linalg.norm(ref)


@pytest.mark.parametrize("d", [64, 128])
@pytest.mark.parametrize("B,H,Lq,Lk,causal,keep", [(4, 16, 256, 700, True, 0.02),   # 32 rows per block, few keys of many tiles
                                                   (4, 16, 200, 200, True, 1.0),    # ... every key of the domain
                                                   (5, 16, 33, 1030, False, 0.01),  # 8 rows: most blocks keep less than a batch
                                                   (9, 16, 40, 129, False, 0.5)])   # 16 rows, one key in a tile of its own
def test_fp32_forward_batches_of_kept_keys(ap, d, B, H, Lq, Lk, causal, keep):
    """Keys kept by a block of rows, gathered from several tiles into batches: sparse and dense lists, partial batches."""
    w = W["tiny"].scaled(B=B, H=H, Lq=Lq, Lk=Lk, d=d, dtype="f32")
    mask = inputs.random_mask(H, Lq, Lk, keep, seed=508, empty_rows=(5,), causal=causal)
    mask[:, :, -1] = mask[:, :, -2]
    q, k, v = inputs.eval_qkv(w)
    tiles = ap.Tiles(H, Lq, Lk)
    ap.ap_mask_to_tiles(mask.cuda(), tiles)
    out = ap.ap_sparse_attention_fwd(q.cuda(), k.cuda(), v.cuda(), tiles, torch.full_like(q, float("nan"), device="cuda"))
    assert ap.ap_device_status() == ap.AP_OK
    ref = orc.attention_fwd(inputs.widen(q), inputs.widen(k), inputs.widen(v), mask.numpy())
    pu.assert_close_attention(out, ref, "f32", str((B, H, Lq, Lk)))
    assert np.all(out[:, :, 5].cpu().numpy() == 0.0)


@pytest.mark.parametrize("bad", [float("inf"), float("nan")])
def test_fp32_forward_pruned_values_are_not_looked_at(ap, bad):
    """A value row of infinities or NaNs reaches the queries that keep its key and no other."""
    w = W["tiny"].scaled(B=2, H=2, Lq=70, Lk=200, d=64, dtype="f32")
    mask = inputs.random_mask(w.H, w.Lq, w.Lk, 0.3, seed=509)
    mask[:, ::2, 150] = 1
    mask[:, 1::2, 150] = 0
    q, k, v = inputs.eval_qkv(w)
    tiles = ap.Tiles(w.H, w.Lq, w.Lk)
    ap.ap_mask_to_tiles(mask.cuda(), tiles)
    ref = orc.attention_fwd(inputs.widen(q), inputs.widen(k), inputs.widen(v), mask.numpy())
    v = v.clone()
    v[:, :, 150] = bad
    out = ap.ap_sparse_attention_fwd(q.cuda(), k.cuda(), v.cuda(), tiles)
    assert ap.ap_device_status() == ap.AP_OK
    assert not torch.isfinite(out[:, :, ::2]).any()
    pu.assert_close_attention(out[:, :, 1::2].contiguous(), ref[:, :, 1::2], "f32")


@pytest.mark.parametrize("B,H,Lq,Lk", [(33, 2, 130, 130),    # eight softmax warps, rows added by entry, chunks
                                       (35, 1, 200, 132),    # ... rows with a tensor map
                                       (150, 12, 64, 64),    # more samples than one wave of CTAs takes: a second launch
                                       (20, 160, 33, 36)])   # more (head, query tile) pairs than SMs
def test_accumulate_many_samples(ap, B, H, Lq, Lk):
    """More samples than a CTA of sixteen softmax warps holds the statistics of."""
    w = W["tiny"].scaled(B=B, H=H, Lq=Lq, Lk=Lk, d=64, dtype="bf16", causal=False)
    bias = inputs.calib_bias(w)
    acc = pu.gpu_accumulate(ap, w, 1, bias.cuda())
    assert ap.ap_device_status() == ap.AP_OK
    assert torch.equal(acc, pu.gpu_accumulate(ap, w, 1, bias.cuda()))
    want = pu.oracle_accumulate(w, 1, bias)
    tol = tp._acc_tolerance(w.dtype)
    np.testing.assert_allclose(acc.cpu().numpy(), want, rtol=tol["rtol"], atol=tol["atol"] * B)


@pytest.mark.parametrize("dtype,d", [("bf16", 64), ("f16", 128)])
@pytest.mark.parametrize("B", [1, 60])     # one CTA per SM at d = 64, or two
@pytest.mark.parametrize("keep", [0.3, 1.0])
def test_entmax_forward_dense_rows(ap, dtype, d, B, keep):
    """Rows with many kept, spread-out entries: the threshold is raised by a chunk's own sums, and some lists overflow."""
    w = W["tiny"].scaled(B=B, H=1, Lq=260, Lk=700 if B == 1 else 300, d=d, dtype=dtype)
    mask = inputs.random_mask(1, w.Lq, w.Lk, keep, seed=511, empty_rows=(9,))
    tp._entmax_fwd_case(ap, w, mask)


def test_build_mask_more_tiles_than_bitmap_words_in_32_bits(ap):
    """2^23 tiles hold 2^32 bitmap words: the entries that the select adds to the bitmaps of the last heads stay with them."""
    H, Lk, k = 1030, 1 << 20, 20
    acc = torch.rand((H, 1, Lk), generator=torch.Generator(device="cuda").manual_seed(510), device="cuda")
    tiles = ap.Tiles(H, 1, Lk, cap=1 << 15)
    ap.ap_build_mask(acc, k / Lk, False, False, tiles=tiles)
    assert ap.ap_device_status() == ap.AP_OK
    row_ptr = tiles.row_ptr.cpu().numpy()
    for h in (0, 3, 1023, 1024, H - 1):
        cols = []
        for t in range(row_ptr[h], row_ptr[h + 1]):
            words = tiles.bitmap[t].cpu().numpy().view(np.uint32)
            assert not words[1:].any()
            bits = np.unpackbits(words[0].view(np.uint8), bitorder="little")
            cols += [int(tiles.col_idx[t]) * 128 + int(c) for c in np.flatnonzero(bits)]
        assert len(cols) == k
        got = acc[h, 0, torch.tensor(cols, device="cuda")].sort(descending=True).values
        assert torch.equal(got, acc[h, 0].topk(k).values)


@pytest.mark.parametrize("dtype", ["bf16", "f16"])
@pytest.mark.parametrize("entry", ["ap_accumulate_attention", "ap_accumulate_attention_entmax15"])
def test_averages_repeat_bit_for_bit(ap, entry, dtype):
    """Three samples and two key tiles: the shape at which the bias tile of the next key tile, already in L2, arrives soonest
    after the threads have handed its place back.  The average was wrong in three of a thousand calls where the copy was not held
    back until their reads were over (a few entries of the first 32 columns, whose reads are the last ones under way)."""
    w = W["s2s_cross"].scaled(B=3, H=2, dtype=dtype)
    bias = inputs.calib_bias(w).cuda()
    q, k = (t.cuda() for t in inputs.calib_qk(w, 0))
    add = getattr(ap, entry)
    want = torch.zeros((w.H, w.Lq, w.Lk), dtype=torch.float32, device="cuda")
    add(want, q, k, bias, causal=w.causal)
    differ = torch.zeros((), dtype=torch.int64, device="cuda")
    for _ in range(3000):
        acc = torch.zeros_like(want)
        add(acc, q, k, bias, causal=w.causal)
        differ += (acc != want).any()
    assert ap.ap_device_status() == ap.AP_OK
    assert int(differ) == 0


@pytest.mark.parametrize("H,Lq,Lk,causal", [(8, 1280, 1280, True), (8, 1281, 1284, True),   # 440 and 528 tiles: 444 are held in shared memory
                                            (1, 384, 18944, False), (1, 385, 18944, False),  # 444 and 592
                                            (127, 40, 50, False), (129, 33, 130, True),     # selections a CTA has several of; too many
                                            (3, 130, 259, True), (1, 1, 1, False), (5, 257, 129, False)])
@pytest.mark.parametrize("rule", ["head", "layer", "ties"])
@pytest.mark.parametrize("distinct", [True, False])
def test_build_mask_held_in_shared_memory(ap, H, Lq, Lk, causal, rule, distinct):
    """The largest inputs that are held and the smallest that are not, ragged edges, rows that start anywhere, a CTA with units of
    several selections; thresholds among many equal values (index digits) and among distinct ones."""
    g = torch.Generator().manual_seed(509 + H)
    acc = torch.rand((H, Lq, Lk), generator=g)
    if not distinct:
        acc = (acc * 7).floor() / 7
    keep, diag = 0.23, causal
    mask = torch.full(acc.shape, 7, dtype=torch.uint8, device="cuda")
    nnz = torch.full((H,), -1, dtype=torch.int64, device="cuda")
    tiles = ap.Tiles(H, Lq, Lk)
    if rule == "ties":
        ap.ap_build_mask_ex(acc.cuda(), keep, causal, diag, ap.AP_MASK_KEEP_TIES, mask, tiles, nnz)
        want, want_nnz = orc.build_mask_ties(acc.numpy(), keep, causal, diag)
    else:
        (ap.ap_build_mask_layer if rule == "layer" else ap.ap_build_mask)(acc.cuda(), keep, causal, diag, mask, tiles, nnz)
        want, want_nnz = (orc.build_mask_layer if rule == "layer" else orc.build_mask)(acc.numpy(), keep, causal, diag)
    assert ap.ap_device_status() == ap.AP_OK
    assert np.array_equal(mask.cpu().numpy(), want)
    assert np.array_equal(nnz.cpu().numpy(), want_nnz)
    pu.assert_tiles_equal(tiles.to_host(), orc.mask_to_tiles(want))


@pytest.mark.parametrize("H,Lq,Lk", [(128, 129, 200), (57, 300, 300),       # 512 and 513 tiles
                                     (300, 513, 600),                       # 1500 list rows: sums are carried from 1024 to the next
                                     (8192, 1, 512), (2731, 8, 1500),    # 32768 and 32772 tiles; the most list rows
                                     (8193, 1, 130), (8, 1, 262400)])    # more list rows; 2050 tiles to a row
def test_list_of_every_size(ap, H, Lq, Lk):
    """The list of a mask, at the limits between the ways of writing it; some rows and tiles are empty."""
    g = torch.Generator().manual_seed(631 + H)
    acc = torch.rand((H, Lq, Lk), generator=g)
    acc[:, :, (Lk // 256) * 128:] *= 0.4  # below the threshold
    mask = torch.empty(acc.shape, dtype=torch.uint8, device="cuda")
    tiles = ap.Tiles(H, Lq, Lk)
    ap.ap_build_mask(acc.cuda(), 0.03, False, False, mask, tiles)
    assert ap.ap_device_status() == ap.AP_OK
    want, _ = orc.build_mask(acc.numpy(), 0.03, False, False)
    assert np.array_equal(mask.cpu().numpy(), want)
    pu.assert_tiles_equal(tiles.to_host(), orc.mask_to_tiles(want))
