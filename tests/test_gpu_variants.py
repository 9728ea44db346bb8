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
