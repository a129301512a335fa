"""Small attention launches, whose tiles are planned in the kernel and shared among the CTAs of a cluster: parts
without a key step, tiles without any, a ragged last block and tile, lists with wrong entries, dense calls, and
sizes on both sides of the rules (1, 2 or 4 CTAs a tile; more tiles than SMs)."""
import numpy as np
import pytest
import torch

from paper_2605_14513_b200 import inputs

from parity import check_attention, to_np

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("block", [64, 128])
@pytest.mark.parametrize("B,H,N", [
    (1, 1, 1),       # one row
    (1, 2, 130),     # one key step a part is too few: not shared
    (2, 1, 512),     # dense: two CTAs a tile
    (1, 2, 2045),    # 32 tiles: four CTAs
    (1, 4, 1029),    # 36 tiles: two
    (1, 65, 255),    # 130 tiles: not shared
    (1, 75, 255),    # 150 tiles: planned by a kernel of its own
])
def test_shared_tiles(oracle, block, B, H, N):
    from paper_2605_14513_b200 import heart

    rs = np.random.RandomState(block + B * H * N)
    g = torch.Generator("cuda").manual_seed(H * N)
    Q, K, V = (torch.randn((B, H, N, 128), generator=g, device="cuda").to(torch.bfloat16) for _ in range(3))
    cfg, nb, R = heart.make_config(B, H, N, block), heart.n_blocks(N, block), B * H
    idx, cnt = np.full((R, nb, nb), -1, np.int32), np.zeros((R, nb), np.int32)
    for r in range(R):
        for I in range(nb):
            sel = rs.permutation(nb)[: rs.choice([0, 1, rs.randint(0, nb + 1), nb])]
            cnt[r, I] = len(sel)
            idx[r, I, : len(sel)] = sel
    ws = heart.new_workspace(cfg)
    every = np.broadcast_to(np.arange(nb, dtype=np.int32), (R, nb, nb)).copy(), np.full((R, nb), nb, np.int32)
    for dense in (False, True):
        O = torch.full_like(Q, float("nan"))
        lse = torch.full((R, N), float("nan"), device="cuda")
        if dense:
            dense_cfg = heart.make_config(B, H, N, block, flags=heart.FORCE_DENSE)
            heart.heart_block_sparse_attn(dense_cfg, Q, K, V, None, None, O, ws, lse=lse)
        else:
            heart.heart_block_sparse_attn(cfg, Q, K, V, torch.from_numpy(idx).cuda(), torch.from_numpy(cnt).cuda(), O, ws, lse=lse)
        assert heart.heart_get_status(ws) == 0
        ref, lse_ref = oracle.block_sparse_attn(*(inputs.bits(t) for t in (Q, K, V)), block, *(every if dense else (idx, cnt)), want_lse=True)
        check_attention(to_np(O.float()).astype(np.float64).reshape(R, N, 128), np.asarray(ref).reshape(R, N, 128))
        got, lse_ref = to_np(lse).reshape(R, N), np.asarray(lse_ref).reshape(R, N)
        assert np.array_equal(np.isneginf(got), np.isneginf(lse_ref))
        fin = np.isfinite(lse_ref)
        # fp32 accumulation of bf16-rounded weights (2^-9 relative each) in the sum behind the logarithm
        assert np.allclose(got[fin], lse_ref[fin], rtol=0, atol=2.0 ** -8)
    idx[0, 0, 0], cnt[0, 0] = nb, max(cnt[0, 0], 1)  # a block that does not exist: skipped, reported
    heart.heart_block_sparse_attn(cfg, Q, K, V, torch.from_numpy(idx).cuda(), torch.from_numpy(cnt).cuda(), O, ws)
    assert heart.heart_get_status(ws) == heart.ERR_DEVICE_CHECK
