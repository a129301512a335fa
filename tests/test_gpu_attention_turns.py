"""How the two softmax warpgroups share the steps of one tile after the other: tiles of 0 to 7 key steps in every order, so that either
warpgroup has a tile's last step and writes the tile before, in layouts whose rows lie between rows of something else (the output
leaves by bulk copies of 32 rows), and the same bits on every run and for every order of the tiles."""
import numpy as np
import pytest
import torch

from paper_2605_14513_b200 import inputs

from parity import check_attention, to_np

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("block", [64, 128])
@pytest.mark.parametrize("H,N,most", [
    (90, 128 * 7 - 31, 7),  # 630 tiles: four or five a CTA; the last rows of a head fill no copy
    (110, 128 * 7 - 31, 7), # 770: short tiles are written at once, the others behind a step of the next one
    (400, 128 + 33, 2),     # tiles of one and two steps only: the roles change with every tile
    (149, 120, 1),          # one tile more than CTAs
    (2, 4500, 36),          # 72 tiles, a pair of CTAs each
    (24, 340, 3),           # 72 tiles of few steps: a CTA each
])
def test_turns(oracle, block, H, N, most):
    from paper_2605_14513_b200 import heart

    rs = np.random.RandomState(block + H + N)
    g = torch.Generator("cuda").manual_seed(H * N)
    Q, K, V = (torch.randn((1, N, H, 128), generator=g, device="cuda").to(torch.bfloat16).permute(0, 2, 1, 3) for _ in range(3))
    nb = heart.n_blocks(N, block)
    idx, cnt = np.full((H, nb, nb), -1, np.int32), np.zeros((H, nb), np.int32)
    for r in range(H):
        for I in range(nb):
            sel = rs.permutation(nb)[: rs.randint(0, min(nb, most * 128 // block) + 1)]
            cnt[r, I] = len(sel)
            idx[r, I, : len(sel)] = sel
    lists = torch.from_numpy(idx).cuda(), torch.from_numpy(cnt).cuda()
    cfg = heart.config_for(Q, block)
    ws = heart.new_workspace(cfg)
    ref, lse_ref = oracle.block_sparse_attn(*(inputs.bits(t) for t in (Q, K, V)), block, idx, cnt, want_lse=True)
    first = None
    for _ in range(3):
        whole = torch.full((1, N + 2, H, 128), 7.0, device="cuda", dtype=torch.bfloat16)  # a row of something else on both sides
        O = whole[:, 1:-1].permute(0, 2, 1, 3)
        lse = torch.full((H, N), float("nan"), device="cuda")
        heart.heart_block_sparse_attn(cfg, Q, K, V, *lists, O, ws, lse=lse)
        assert heart.heart_get_status(ws) == 0
        assert (whole[:, 0] == 7.0).all() and (whole[:, -1] == 7.0).all()
        if first is None:
            first = O.clone(), lse
            check_attention(to_np(O.float()).astype(np.float64).reshape(H, N, 128), ref)
            got, fin = to_np(lse), np.isfinite(lse_ref)
            assert np.array_equal(np.isneginf(got), np.isneginf(lse_ref))
            # fp32 accumulation of bf16-rounded weights (2^-9 relative each) in the sum behind the logarithm
            assert np.allclose(got[fin], lse_ref[fin], rtol=0, atol=2.0 ** -8)
        assert torch.equal(O.contiguous().view(torch.int16), first[0].contiguous().view(torch.int16)) and torch.equal(lse, first[1])


@pytest.mark.parametrize("block", [64, 128])
@pytest.mark.parametrize("H,N,steps", [
    (3, 128, 1), (5, 77, 1), (20, 500, 1), (60, 300, 1),
    (2, 2045, 1), (2, 2045, 3), (2, 2045, 4),  # launched as clusters of four; shared from four steps on
    (4, 1029, 2), (4, 1029, 3), (4, 1029, 4),  # of two
    (2, 4500, 3), (2, 4500, 5),                # 72 tiles, pairs
])
def test_tiles_of_a_few_steps_in_small_launches(oracle, block, H, N, steps):
    """With one step, the warpgroup without it writes the tile and its log-sum-exps straight away, by what it has just noted of the
    tile; up to three, one CTA of a cluster takes all of them."""
    from paper_2605_14513_b200 import heart

    g = torch.Generator("cuda").manual_seed(H * N + block)
    Q, K, V = (torch.randn((1, H, N, 128), generator=g, device="cuda").to(torch.bfloat16) for _ in range(3))
    nb, per = heart.n_blocks(N, block), 128 // block
    idx, cnt = np.full((H, nb, nb), -1, np.int32), np.full((H, nb), min(nb, steps * per), np.int32)
    first = per * (np.arange(H)[:, None] + np.arange(nb) // per)  # the query blocks of a tile list the same key blocks
    for k in range(cnt[0, 0]):
        idx[:, :, k] = (first + k) % nb
    cfg = heart.config_for(Q, block)
    ws, O, lse = heart.new_workspace(cfg), torch.full_like(Q, float("nan")), torch.full((H, N), float("nan"), device="cuda")
    heart.heart_block_sparse_attn(cfg, Q, K, V, torch.from_numpy(idx).cuda(), torch.from_numpy(cnt).cuda(), O, ws, lse=lse)
    assert heart.heart_get_status(ws) == 0
    ref, lse_ref = oracle.block_sparse_attn(*(inputs.bits(t) for t in (Q, K, V)), block, idx, cnt, want_lse=True)
    check_attention(to_np(O.float()).astype(np.float64).reshape(H, N, 128), ref)
    # fp32 accumulation of bf16-rounded weights (2^-9 relative each) in the sum behind the logarithm
    assert np.allclose(to_np(lse), lse_ref, rtol=0, atol=2.0 ** -8)


@pytest.mark.parametrize("H,N", [(2, 1), (1, 130), (2, 2045), (60, 700), (1, 9000), (1, 9473)])  # shared tiles (71: pairs; 75: a CTA each), several; ragged blocks
def test_dense_calls_do_not_depend_on_the_block(H, N):
    from paper_2605_14513_b200 import heart

    g = torch.Generator("cuda").manual_seed(H * N)
    Q, K, V = (torch.randn((1, H, N, 128), generator=g, device="cuda").to(torch.bfloat16) for _ in range(3))
    outs = []
    for block in (64, 128):
        cfg = heart.make_config(1, H, N, block, flags=heart.FORCE_DENSE)
        ws, O, lse = heart.new_workspace(cfg), torch.full_like(Q, float("nan")), torch.full((H, N), float("nan"), device="cuda")
        heart.heart_block_sparse_attn(cfg, Q, K, V, None, None, O, ws, lse=lse)
        assert heart.heart_get_status(ws) == 0
        outs.append((O, lse))
    assert torch.equal(outs[0][0].view(torch.int16), outs[1][0].view(torch.int16)) and torch.equal(outs[0][1], outs[1][1])
    ref = torch.nn.functional.scaled_dot_product_attention(Q.double(), K.double(), V.double())
    check_attention(to_np(outs[0][0].float()).astype(np.float64).reshape(H, N, 128), to_np(ref).reshape(H, N, 128))


@pytest.mark.parametrize("block", [64, 128])
@pytest.mark.parametrize("dense", [False, True])
@pytest.mark.parametrize("H,N", [(40, 420), (16, 1300)])  # 160 and 176 tiles in all, 8 to 12 in a group of heads
def test_head_groups_give_the_bits_of_the_whole(block, dense, H, N):
    """heart_step_host runs its heads in groups, of a tile per CTA here, heart_step all of them with several tiles per CTA: the order
    of a row's sums goes by the tiles of all heads, so the outputs are equal bit for bit."""
    from paper_2605_14513_b200 import heart

    g = torch.Generator("cuda").manual_seed(H * N + block)
    Q, K, V = (torch.randn((1, H, N, 128), generator=g, device="cuda").to(torch.bfloat16) for _ in range(3))
    cfg = heart.make_config(1, H, N, block, flags=heart.FORCE_DENSE if dense else 0)
    delta = torch.full((H,), -1.0, dtype=torch.float64, device="cuda")
    tau = torch.linspace(0.3, 0.95, H, dtype=torch.float64, device="cuda")
    whole, groups, ws, ws_host = heart.State(cfg), heart.State(cfg), heart.new_workspace(cfg), heart.new_workspace(cfg)
    O = torch.full_like(Q, float("nan"))
    heart.heart_step(cfg, Q, K, V, delta, tau, whole, O, ws)
    host = [x.cpu().pin_memory() for x in (Q, K, V)]
    O_host = torch.full(Q.shape, float("nan"), dtype=torch.bfloat16).pin_memory()
    heart.heart_step_host(cfg, *host, delta, tau, groups, O_host, tuple(torch.empty_like(Q) for _ in range(4)), ws_host)
    assert heart.heart_get_status(ws) == 0 and heart.heart_get_status(ws_host) == 0
    assert not O.isnan().any()
    assert torch.equal(O.cpu().view(torch.int16), O_host.view(torch.int16))
