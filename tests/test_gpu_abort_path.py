"""The attention kernel's time-out path, taken once under test without faulting or hanging anything.

Every wait in the kernel is bounded; when one runs out the CTA raises an abort flag, its roles
drain (copies and tensor-core products in flight are waited for, with a bound), tensor memory is
released, the CTA exits and the workspace's status word reports HEART_ERR_DEVICE_CHECK.  The
test-hook build of the library (same sources, HEART_TEST_HOOKS, a wait limit of 2e6 clocks) has one
reserved flag bit that makes the V producer of CTA 0 leave out one copy -- neither the byte count is
announced nor the copy issued -- so the waits that depend on that tile run out after about a
millisecond; another bit keeps a CTA's part of a shared tile from the other CTAs of its cluster, a third leaves out the K copy of the
first key step of CTA 0's second tile.  Nothing traps and nothing waits without a bound.
"""
import time

import numpy as np
import pytest
import torch

from paper_2605_14513_b200 import build as heart_build
from paper_2605_14513_b200 import inputs

pytestmark = pytest.mark.gpu

TEST_SKIP_V = 0x80000000
TEST_SKIP_PARTS = 0x40000000
TEST_SKIP_K = 0x20000000


def dense_attention(h, flags, Q, K, V, wl):
    cfg = h.make_config(wl.B, wl.H, wl.N, wl.block, flags=h.FORCE_DENSE | flags)
    ws = h.new_workspace(cfg)
    O = torch.full_like(Q, float("nan"))
    t0 = time.perf_counter()
    h.heart_block_sparse_attn(cfg, Q, K, V, None, None, O, ws)
    status = h.heart_get_status(ws)  # synchronises
    return O, status, time.perf_counter() - t0, (cfg, ws)


def test_a_wait_that_runs_out_is_reported_and_the_context_stays_usable():
    from paper_2605_14513_b200 import heart as h

    assert torch.cuda.is_available()
    product = h.lib()
    hooks = h.load(heart_build.build_test_hooks())
    wl = inputs.small_workload(H=2, grid=(3, 10, 14), block=64, seed=41)  # N = 420: 4 query tiles a head, 7 key steps
    Q, K, V = inputs.Sequence(wl, "cuda").bf16()
    try:
        h._lib = hooks
        O_ref, status, _, _ = dense_attention(h, 0, Q, K, V, wl)
        assert status == 0
        O_bad, status, seconds, (cfg, ws) = dense_attention(h, TEST_SKIP_V, Q, K, V, wl)
        assert status == h.ERR_DEVICE_CHECK          # the wait ran out and said so
        assert seconds < 5.0                          # ... after milliseconds, not the product's 2 s limit
        assert h.heart_get_status(ws) == 0            # the status word is cleared by the read
        # CTA 0 (head 0, query rows 0..127) gave up without writing; every other tile is complete
        ref, bad = O_ref.view(wl.R, wl.N, wl.D), O_bad.view(wl.R, wl.N, wl.D)
        assert torch.isnan(bad[0, :128].float()).all()
        assert torch.equal(bad[0, 128:].view(torch.int16), ref[0, 128:].view(torch.int16))
        assert torch.equal(bad[1].view(torch.int16), ref[1].view(torch.int16))
        # the same workspace and the same context serve a normal call right after, bit for bit
        cfg.flags = h.FORCE_DENSE
        O_again = torch.full_like(Q, float("nan"))
        h.heart_block_sparse_attn(cfg, Q, K, V, None, None, O_again, ws)
        assert h.heart_get_status(ws) == 0
        assert torch.equal(O_again.view(torch.int16), O_ref.view(torch.int16))
    finally:
        h._lib = product
    # the product library has no such hook: the reserved bit changes nothing there
    O_prod, status, _, _ = dense_attention(h, TEST_SKIP_V, Q, K, V, wl)
    assert status == 0
    assert torch.equal(O_prod.view(torch.int16), O_ref.view(torch.int16))


@pytest.fixture
def hooks():
    from paper_2605_14513_b200 import heart as h

    product = h.lib()
    h._lib = h.load(heart_build.build_test_hooks())
    yield h
    h._lib = product


@pytest.mark.parametrize("block", [64, 128])
@pytest.mark.parametrize("H,N", [(2, 420), (2, 2045), (80, 257)])  # tiles shared by two CTAs (dense; lists of 4 steps are not) and by four; 240 tiles of 2 or 3 steps for 148 CTAs
def test_other_tiles_are_complete_after_an_abort(hooks, block, H, N):
    h = hooks
    g = torch.Generator("cuda").manual_seed(N)
    Q, K, V = (torch.randn((1, H, N, 128), generator=g, device="cuda").to(torch.bfloat16) for _ in range(3))
    nb, tiles = h.n_blocks(N, block), (N + 127) // 128
    idx = torch.arange(nb, dtype=torch.int32, device="cuda").expand(H, nb, nb).contiguous()
    cnt = torch.full((H, nb), nb, dtype=torch.int32, device="cuda")
    for dense in (True, False):
        cfg = h.make_config(1, H, N, block, flags=h.FORCE_DENSE if dense else 0)
        use = (None, None) if dense else (idx, cnt)
        ws = h.new_workspace(cfg)
        ref, bad, again = (torch.full_like(Q, float("nan")) for _ in range(3))
        h.heart_block_sparse_attn(cfg, Q, K, V, *use, ref, ws)
        assert h.heart_get_status(ws) == 0 and not ref.isnan().any()
        cfg.flags |= TEST_SKIP_V
        t0 = time.perf_counter()
        h.heart_block_sparse_attn(cfg, Q, K, V, *use, bad, ws)
        assert h.heart_get_status(ws) == h.ERR_DEVICE_CHECK
        assert time.perf_counter() - t0 < 5.0
        lost = [(head, t) for head in range(H) for t in range(tiles) if bad[0, head, 128 * t].isnan().any()]
        if H * tiles <= 148 or dense:  # the tiles of CTA 0 are known
            assert lost == [divmod(n, tiles) for n in range(0, H * tiles, 148)]
        else:  # its first one, and the next if that was drawn already
            assert 1 <= len(lost) <= 2
        for head, t in lost:
            assert bad[0, head, 128 * t : 128 * t + 128].isnan().all()
            bad[0, head, 128 * t : 128 * t + 128] = ref[0, head, 128 * t : 128 * t + 128]
        assert torch.equal(bad.view(torch.int16), ref.view(torch.int16))
        cfg.flags &= ~TEST_SKIP_V
        h.heart_block_sparse_attn(cfg, Q, K, V, *use, again, ws)
        assert h.heart_get_status(ws) == 0
        assert torch.equal(again.view(torch.int16), ref.view(torch.int16))


@pytest.mark.parametrize("block", [64, 128])
@pytest.mark.parametrize("H,N", [(4, 1029), (2, 4500)])  # 9 and 36 key steps: two CTAs a tile, lists too
def test_other_tiles_are_complete_after_an_abort_in_a_pair(hooks, block, H, N):
    test_other_tiles_are_complete_after_an_abort(hooks, block, H, N)


@pytest.mark.parametrize("block", [64, 128])
@pytest.mark.parametrize("H,N", [(200, 257), (80, 1000), (600, 128), (300, 256), (400, 256)])  # four tiles a CTA and more, of 3, 8, 1, 2 and 2 steps
def test_a_finished_tile_survives_the_abort_of_the_next(hooks, block, H, N):
    """The products of CTA 0's first tile are complete when the wait for its second tile's first scores runs out: the first
    tile's output and log-sum-exps are there, the second tile is the one that is lost."""
    h = hooks
    g = torch.Generator("cuda").manual_seed(N + block)
    Q, K, V = (torch.randn((1, H, N, 128), generator=g, device="cuda").to(torch.bfloat16) for _ in range(3))
    nb, tiles = h.n_blocks(N, block), (N + 127) // 128
    idx = torch.arange(nb, dtype=torch.int32, device="cuda").expand(H, nb, nb).contiguous()
    cnt = torch.full((H, nb), nb, dtype=torch.int32, device="cuda")
    for dense in (True, False):
        cfg = h.make_config(1, H, N, block, flags=h.FORCE_DENSE if dense else 0)
        use = (None, None) if dense else (idx, cnt)
        ws = h.new_workspace(cfg)
        ref, bad = (torch.full_like(Q, float("nan")) for _ in range(2))
        lse_ref, lse_bad = (torch.full((H, N), float("nan"), device="cuda") for _ in range(2))
        h.heart_block_sparse_attn(cfg, Q, K, V, *use, ref, ws, lse=lse_ref)
        assert h.heart_get_status(ws) == 0 and not ref.isnan().any()
        cfg.flags |= TEST_SKIP_K
        t0 = time.perf_counter()
        h.heart_block_sparse_attn(cfg, Q, K, V, *use, bad, ws, lse=lse_bad)
        assert h.heart_get_status(ws) == h.ERR_DEVICE_CHECK
        assert time.perf_counter() - t0 < 5.0
        lost = [(head, t) for head in range(H) for t in range(tiles) if bad[0, head, 128 * t].isnan().any()]
        if dense:  # dealt in turn
            assert lost == [divmod(n, tiles) for n in range(148, H * tiles, 148)]
        else:  # its second tile, and those drawn behind it already
            assert 1 <= len(lost) <= 3
        for head, t in lost:
            rows = slice(128 * t, 128 * t + 128)
            assert bad[0, head, rows].isnan().all() and lse_bad[head, rows].isnan().all()
            bad[0, head, rows], lse_bad[head, rows] = ref[0, head, rows], lse_ref[head, rows]
        assert torch.equal(bad.view(torch.int16), ref.view(torch.int16)) and torch.equal(lse_bad, lse_ref)
        again = torch.full_like(Q, float("nan"))
        cfg.flags &= ~TEST_SKIP_K
        h.heart_block_sparse_attn(cfg, Q, K, V, *use, again, ws)
        assert h.heart_get_status(ws) == 0
        assert torch.equal(again.view(torch.int16), ref.view(torch.int16))


@pytest.mark.parametrize("block", [64, 128])
@pytest.mark.parametrize("N,split", [(420, 2), (2045, 4)])
def test_a_part_that_never_arrives(hooks, block, N, split):
    """The CTAs that wait for it report it and leave all of their rows of the tile alone; its own rows, for which it has the
    other parts, and the other tiles are complete."""
    h, H = hooks, 2
    g = torch.Generator("cuda").manual_seed(N + block)
    Q, K, V = (torch.randn((1, H, N, 128), generator=g, device="cuda").to(torch.bfloat16) for _ in range(3))
    cfg = h.make_config(1, H, N, block, flags=h.FORCE_DENSE)
    ws = h.new_workspace(cfg)
    ref, bad, again = (torch.full_like(Q, float("nan")) for _ in range(3))
    h.heart_block_sparse_attn(cfg, Q, K, V, None, None, ref, ws)
    assert h.heart_get_status(ws) == 0
    cfg.flags |= TEST_SKIP_PARTS
    t0 = time.perf_counter()
    h.heart_block_sparse_attn(cfg, Q, K, V, None, None, bad, ws)
    assert h.heart_get_status(ws) == h.ERR_DEVICE_CHECK
    assert time.perf_counter() - t0 < 5.0
    rows = 128 // split
    for r in range(split):
        part = bad[0, 0, r * rows : (r + 1) * rows]
        if r != 1:
            assert part.isnan().all()
            part.copy_(ref[0, 0, r * rows : (r + 1) * rows])
    assert torch.equal(bad.view(torch.int16), ref.view(torch.int16))
    cfg.flags &= ~TEST_SKIP_PARTS
    h.heart_block_sparse_attn(cfg, Q, K, V, None, None, again, ws)
    assert h.heart_get_status(ws) == 0
    assert torch.equal(again.view(torch.int16), ref.view(torch.int16))


@pytest.mark.parametrize("block", [64, 128])
@pytest.mark.parametrize("H,N", [(2, 600), (100, 600), (3, 9000)])  # a tile a pair; more tiles than pairs; 9 tiles a head
def test_antidiagonal_pair_that_gives_up(hooks, block, H, N):
    h = hooks
    g = torch.Generator("cuda").manual_seed(N)
    Q, K = (torch.randn((1, H, N, 128), generator=g, device="cuda").to(torch.bfloat16) for _ in range(2))
    cfg = h.make_config(1, H, N, block, flags=h.ESTIMATOR_ANTIDIAG)
    tau = torch.full((H,), 0.9, dtype=torch.float64, device="cuda")
    ws, ref, bad, again = h.new_workspace(cfg), h.State(cfg), h.State(cfg), h.State(cfg)
    h.heart_predict_mask(cfg, Q, K, tau, ref, ws)
    assert h.heart_get_status(ws) == 0
    cfg.flags |= TEST_SKIP_V
    t0 = time.perf_counter()
    h.heart_predict_mask(cfg, Q, K, tau, bad, ws)
    assert h.heart_get_status(ws) == h.ERR_DEVICE_CHECK
    assert time.perf_counter() - t0 < 5.0
    cfg.flags &= ~TEST_SKIP_V
    h.heart_predict_mask(cfg, Q, K, tau, again, ws)
    assert h.heart_get_status(ws) == 0
    assert torch.equal(again.kv_cnt, ref.kv_cnt) and torch.equal(again.mask_bits, ref.mask_bits)
