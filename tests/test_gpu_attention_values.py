"""Attention on values at the edges of what the inputs can hold, in launches on both sides of the rules that pick a
path (1, 2 or 4 CTAs a tile; tiles planned in the kernel or by one of their own; dense)."""
import numpy as np
import pytest
import torch

from paper_2605_14513_b200 import inputs

from parity import check_attention, to_np

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


def staircase(rs, H, N, v_scale=1.0):
    """Q, K, V whose rows see their maximum climb and fall from one key step to the next by amounts on both sides of
    those at which the kernel moves a row's reference, in 64 patterns a head that are dealt to the rows at random.
    Pattern c of a row is read off dims c and c + 64 of the keys (a coarse and a fine part of the logit)."""
    levels = rs.uniform(-60, 60, (H, 64, 1)) + np.cumsum(
        rs.choice([-40, -5, -1, 0, 1, 2, 3, 5, 7, 9, 29, 31, 33, 61], (H, 64, (N + 63) // 64),
                  p=[.04, .08, .1, .1, .1, .1, .1, .08, .05, .05, .05, .05, .05, .05]), axis=2)
    logit = (np.repeat(levels, 64, axis=2)[:, :, :N] - rs.uniform(0, 3, (H, 64, N))) * np.log(2.0)
    logit = torch.from_numpy(np.moveaxis(logit, 1, 2).copy())  # [H, N, 64]
    coarse = logit.to(torch.bfloat16)
    K = torch.cat([coarse, (logit - coarse.double()).to(torch.bfloat16)], dim=2)
    pattern = torch.from_numpy(rs.randint(0, 64, (H, N, 1)))
    Q = torch.zeros((H, N, 128), dtype=torch.bfloat16)
    Q.scatter_(2, pattern, 1.0)
    Q.scatter_(2, pattern + 64, 1.0)
    V = (torch.from_numpy(rs.standard_normal((H, N, 128))) * v_scale).to(torch.bfloat16)
    return tuple(x[None].cuda().contiguous() for x in (Q, K, V))


@pytest.mark.parametrize("block", [64, 128])
@pytest.mark.parametrize("v_scale", [1.0, 2.0 ** 100])
@pytest.mark.parametrize("H,N", [(2, 2045), (4, 1029), (8, 1000), (12, 1700)])
def test_row_maxima_that_climb_from_step_to_step(oracle, block, v_scale, H, N):
    """Contributions from before a move of the reference still count after it (a maximum that climbs by 31 and then by
    2 powers of two, say), the moves fall on even and odd key steps of rows next to each other, and values of V near
    the top of the range do not overflow on the way: a result is a mean of them."""
    from paper_2605_14513_b200 import heart

    rs = np.random.RandomState(H * N + block)
    Q, K, V = staircase(rs, H, N, v_scale)
    nb = heart.n_blocks(N, block)
    idx, cnt = np.zeros((H, nb, nb), np.int32), np.zeros((H, nb), np.int32)
    for r in range(H):
        for I in range(nb):
            sel = np.sort(rs.permutation(nb)[: rs.choice([nb, nb - 1, (nb + 1) // 2])])
            cnt[r, I], idx[r, I, : len(sel)] = len(sel), sel
    O, lse = attend(heart, heart.make_config(1, H, N, block, scale=1.0), Q, K, V, (torch.from_numpy(idx).cuda(), torch.from_numpy(cnt).cuda()))
    ref, lse_ref = oracle.block_sparse_attn(*(inputs.bits(t) for t in (Q, K, V)), block, idx, cnt, scale=1.0, want_lse=True)
    ref, lse_ref = np.asarray(ref).reshape(H, N, 128), np.asarray(lse_ref).reshape(H, N)
    check_attention(O.astype(np.float64) / v_scale, ref / v_scale)
    # fp32 scores up to 2^10 (2^-14) and bf16-rounded weights (2^-9 relative each) in the sum behind the logarithm
    assert np.allclose(lse, lse_ref, rtol=0, atol=2.0 ** -8)
