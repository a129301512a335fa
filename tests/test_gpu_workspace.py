"""What a call leaves alone in the workspace: a mask prediction for one layer may run on a second stream beside the
attention of another on the same workspace, and so may a dense attention."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


def lists(rs, R, nb, keep):
    idx, cnt = np.zeros((R, nb, nb), np.int32), np.zeros((R, nb), np.int32)
    for r in range(R):
        for I in range(nb):
            sel = np.sort(rs.permutation(nb)[: max(1, int(keep * nb))])
            cnt[r, I], idx[r, I, : len(sel)] = len(sel), sel
    return torch.from_numpy(idx).cuda(), torch.from_numpy(cnt).cuda()


def tensors(H, N, seed, n=3):
    g = torch.Generator("cuda").manual_seed(seed)
    return [torch.randn((1, H, N, 128), generator=g, device="cuda").to(torch.bfloat16) for _ in range(n)]


def changed(ws, before):
    """Bytes that a call wrote, the status words (the first 256 bytes) left out."""
    return (ws != before)[256:]


@pytest.mark.parametrize("block", [64, 128])
@pytest.mark.parametrize("H,N", [(1, 100), (2, 2045), (5, 4100)])
def test_attention_writes_nothing_that_drift_and_mask_prediction_write(block, H, N):
    from paper_2605_14513_b200 import heart

    Q, K, V = tensors(H, N, N)
    cfg = heart.make_config(1, H, N, block)
    idx, cnt = lists(np.random.RandomState(N), H, heart.n_blocks(N, block), 0.4)
    st, tau = heart.State(cfg), torch.full((H,), 0.9, dtype=torch.float64, device="cuda")
    by_attention, by_masks = (torch.zeros(heart.workspace_bytes(cfg) - 256, dtype=torch.bool, device="cuda") for _ in range(2))
    for fill in (0x55, 0xAA):  # a byte that is rewritten as it was shows with the other filling
        ws = torch.full((heart.workspace_bytes(cfg),), fill, dtype=torch.uint8, device="cuda")
        ws[:256] = 0
        before = ws.clone()
        heart.heart_block_sparse_attn(cfg, Q, K, V, idx, cnt, torch.empty_like(Q), ws)
        assert heart.heart_get_status(ws) == 0
        by_attention |= changed(ws, before)
        before = ws.clone()
        heart.heart_drift(cfg, Q, K, tau, st, ws)
        heart.heart_predict_mask(cfg, Q, K, tau, st, ws)
        assert heart.heart_get_status(ws) == 0
        by_masks |= changed(ws, before)
    assert by_masks.any() and not (by_attention & by_masks).any()
    scores = heart.drift_workspace_bytes(cfg) - 256
    assert by_masks[scores:].any() and not by_attention[scores:].any()


@pytest.mark.parametrize("block", [64, 128])
def test_mask_prediction_beside_attention_on_one_workspace(block):
    from paper_2605_14513_b200 import heart

    H, N = 8, 8100
    Q, K, V = tensors(H, N, 1)
    Q2, K2 = tensors(H, N, 2, n=2)
    cfg = heart.make_config(1, H, N, block)
    idx, cnt = lists(np.random.RandomState(0), H, heart.n_blocks(N, block), 0.5)
    tau = torch.full((H,), 0.9, dtype=torch.float64, device="cuda")
    ws, want, st_want = heart.new_workspace(cfg), torch.empty_like(Q), heart.State(cfg)
    heart.heart_block_sparse_attn(cfg, Q, K, V, idx, cnt, want, ws)
    heart.heart_predict_mask(cfg, Q2, K2, tau, st_want, ws)
    torch.cuda.synchronize()
    side = torch.cuda.Stream()
    for _ in range(10):
        O, st = torch.empty_like(Q), heart.State(cfg)
        torch.cuda.synchronize()
        heart.heart_block_sparse_attn(cfg, Q, K, V, idx, cnt, O, ws)
        with torch.cuda.stream(side):
            for _ in range(4):
                heart.heart_predict_mask(cfg, Q2, K2, tau, st, ws)
        torch.cuda.synchronize()
        assert heart.heart_get_status(ws) == 0
        assert torch.equal(O.view(torch.int16), want.view(torch.int16))
        assert torch.equal(st.kv_cnt, st_want.kv_cnt) and torch.equal(st.mask_bits, st_want.mask_bits)


@pytest.mark.parametrize("block", [64, 128])
def test_dense_attention_beside_attention_on_one_workspace(block):
    from paper_2605_14513_b200 import heart

    H, N = 8, 8100
    Q, K, V = tensors(H, N, 3)
    idx, cnt = lists(np.random.RandomState(1), H, heart.n_blocks(N, block), 0.5)
    cfg, dense = heart.make_config(1, H, N, block), heart.make_config(1, H, N, block, flags=heart.FORCE_DENSE)
    ws = heart.new_workspace(cfg)
    want, want_dense = torch.empty_like(Q), torch.empty_like(Q)
    heart.heart_block_sparse_attn(dense, Q, K, V, None, None, want_dense, ws)
    assert not ws.any()  # nothing is kept there, so nothing can be in another call's way
    heart.heart_block_sparse_attn(cfg, Q, K, V, idx, cnt, want, ws)
    torch.cuda.synchronize()
    side = [torch.cuda.Stream() for _ in range(2)]
    for _ in range(5):
        O, dense_out = torch.empty_like(Q), [torch.empty_like(Q) for _ in side]
        torch.cuda.synchronize()
        heart.heart_block_sparse_attn(cfg, Q, K, V, idx, cnt, O, ws)
        for s, out in zip(side, dense_out):
            with torch.cuda.stream(s):
                heart.heart_block_sparse_attn(dense, Q, K, V, None, None, out, ws)
        torch.cuda.synchronize()
        assert heart.heart_get_status(ws) == 0
        assert torch.equal(O.view(torch.int16), want.view(torch.int16))
        assert all(torch.equal(out.view(torch.int16), want_dense.view(torch.int16)) for out in dense_out)
