"""The attention kernel's step lists and tile queue at their edges: odd numbers of listed blocks, key
blocks that only one of a tile's two query blocks lists, the ragged last block in either half of a step,
query blocks without any key block (runs of them longer than the announcement ring), and more tiles than
there are CTAs (148), so that tiles are drawn from the counter."""
import numpy as np
import pytest
import torch

from paper_2605_14513_b200 import inputs

from parity import check_attention, to_np

pytestmark = pytest.mark.gpu


def make_lists(rs, R, nb, kind, block):
    idx, cnt = np.full((R, nb, nb), -1, np.int32), np.zeros((R, nb), np.int32)
    for r in range(R):
        for I in range(nb):
            if kind == "disjoint":  # the two query blocks of a 128-row tile share no key block
                sel = np.arange(I % 2, nb, 2)
            elif kind == "one_sided":  # only one of them lists anything; an odd number, the last block included
                sel = np.arange(nb - (nb - 1) % 2 - 1, nb) if I % 2 else np.empty(0, int)
            elif kind == "empty_runs":  # most heads empty
                sel = np.sort(rs.choice(nb, rs.randint(1, nb + 1), replace=False)) if r % 7 == 0 else np.empty(0, int)
            else:  # random order inside the list, every count from none to all
                sel = rs.permutation(nb)[: rs.randint(0, nb + 1)]
            cnt[r, I] = len(sel)
            idx[r, I, : len(sel)] = sel
    return idx, cnt


@pytest.mark.parametrize("block", [64, 128])
@pytest.mark.parametrize("kind,H,N", [
    ("random", 3, 700),        # 6 tiles: every CTA at most one
    ("random", 110, 330),      # 330 tiles of 3 a head: CTAs draw a second and a third tile; ragged last tile and block
    ("disjoint", 2, 64 * 9 + 5),
    ("one_sided", 2, 64 * 8 - 3),
    ("empty_runs", 160, 257),  # 480 tiles, runs of 18 empty ones
])
def test_lists_and_tile_queue(oracle, block, kind, H, N):
    from paper_2605_14513_b200 import heart

    rs = np.random.RandomState(block + H + N)
    g = torch.Generator("cuda").manual_seed(H * N)
    Q, K, V = (torch.randn((1, H, N, 128), generator=g, device="cuda").to(torch.bfloat16) for _ in range(3))
    cfg = heart.make_config(1, H, N, block)
    nb = heart.n_blocks(N, block)
    idx, cnt = make_lists(rs, H, nb, kind, block)
    O = torch.full_like(Q, float("nan"))
    lse = torch.full((H, N), float("nan"), device="cuda")
    ws = heart.new_workspace(cfg)
    for _ in range(2):  # the second launch starts from the counter that the first one leaves
        heart.heart_block_sparse_attn(cfg, Q, K, V, torch.from_numpy(idx).cuda(), torch.from_numpy(cnt).cuda(), O, ws, lse=lse)
        assert heart.heart_get_status(ws) == 0
        ref, lse_ref = oracle.block_sparse_attn(*(inputs.bits(t) for t in (Q, K, V)), block, idx, cnt, want_lse=True)
        check_attention(to_np(O.float()).astype(np.float64).reshape(H, N, 128), ref)
        got = to_np(lse)
        assert np.array_equal(np.isneginf(got), np.isneginf(lse_ref))
        fin = np.isfinite(lse_ref)
        # fp32 accumulation of bf16-rounded weights (2^-9 relative each) in the sum behind the logarithm
        assert np.allclose(got[fin], lse_ref[fin], rtol=0, atol=2.0 ** -8)
        O.fill_(float("nan"))
