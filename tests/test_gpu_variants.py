"""GPU parity of kernel variants that a rule on sizes chooses, at the sizes where each can go wrong: edges of
its tiles, remainders, the smallest and the largest shapes of its range."""
import numpy as np
import pytest
import torch

from oracle import ap_oracle as orc
from paper_2012_02030_b200 import inputs
from tests import parity_util as pu

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
