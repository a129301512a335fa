"""Attention on values at the edges of what the inputs can hold, in launches on both sides of the rules that pick a
path (1, 2 or 4 CTAs a tile; tiles planned in the kernel or by one of their own; dense)."""
import numpy as np
import pytest
import torch

from parity import to_np

pytestmark = pytest.mark.gpu

# (H, N): four CTAs a tile; two; one; tiles planned by a kernel of their own
SIZES = [(2, 2045), (4, 1029), (65, 255), (75, 255)]


def attend(heart, cfg, Q, K, V, lists=(None, None)):
    O = torch.full_like(Q, 7.0)
    lse = torch.full((cfg.B * cfg.H, cfg.N), 7.0, device="cuda")
    ws = heart.new_workspace(cfg)
    heart.heart_block_sparse_attn(cfg, Q, K, V, *lists, O, ws, lse=lse)
    assert heart.heart_get_status(ws) == 0
    return to_np(O.float())[0], to_np(lse)


@pytest.mark.parametrize("block", [64, 128])
@pytest.mark.parametrize("H,N", SIZES)
def test_a_value_that_is_not_a_number_reaches_the_rows_that_use_it_and_no_others(block, H, N):
    from paper_2605_14513_b200 import heart

    g = torch.Generator("cuda").manual_seed(N)
    Q, K, V = (torch.randn((1, H, N, 128), generator=g, device="cuda").to(torch.bfloat16) for _ in range(3))
    nb = heart.n_blocks(N, block)
    q_row, k_row = 5, N - 3  # the row of Q in head 1, the key in head 0
    idx = np.broadcast_to(np.arange(nb, dtype=np.int32), (H, nb, nb)).copy()
    cnt = np.full((H, nb), nb, np.int32)
    cnt[0, 1::2] = nb - 1  # odd query blocks of head 0 do not list the last key block
    lists = torch.from_numpy(idx).cuda(), torch.from_numpy(cnt).cuda()
    for dense in (False, True):
        cfg = heart.make_config(1, H, N, block, flags=heart.FORCE_DENSE if dense else 0)
        use = (None, None) if dense else lists
        O, lse = attend(heart, cfg, Q, K, V, use)
        Qn, Kn = Q.clone(), K.clone()
        Qn[0, 1, q_row, 17] = float("nan")
        Kn[0, 0, k_row, 90] = float("nan")
        On, lse_n = attend(heart, cfg, Qn, Kn, V, use)
        hit = np.zeros((H, N), bool)
        hit[1, q_row] = True
        hit[0] = True if dense else (np.arange(N) // block) % 2 == 0
        assert np.isnan(On[hit]).all() and not np.isfinite(lse_n[hit]).any()
        assert np.array_equal(On[~hit], O[~hit]) and np.array_equal(lse_n[~hit], lse[~hit])
