"""The layer gate of small steps, which the row kernel applies: below, between and above its limits, in several batch entries with
another outcome each, more heads than the kernel has threads, heads without an anchor, against heart_drift, which has the
gate in its own kernel."""
import pytest
import torch

from test_gpu_small_steps import both_ways

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("B,H,N,block", [(3, 4, 300, 64), (1, 48, 130, 64), (2, 257, 60, 64), (1, 600, 20, 128), (2, 12, 2465, 64), (4, 1, 900, 128)])
def test_gate(B, H, N, block):
    from paper_2605_14513_b200 import heart

    g = torch.Generator("cuda").manual_seed(B * H * N)
    R = B * H
    cfg = heart.make_config(B, H, N, block, gate_lo=0.4, gate_hi=0.6)
    st, calls, ws, calls_ws = heart.State(cfg), heart.State(cfg), heart.new_workspace(cfg), heart.new_workspace(cfg)
    tau = torch.linspace(0.5, 0.95, R, dtype=torch.float64, device="cuda")
    seen = set()
    for step in range(6):
        Q, K, V = (torch.randn((B, H, N, 128), generator=g, device="cuda").to(torch.bfloat16) for _ in range(3))
        # a share of refreshing heads of its own for every batch entry: all reuse, as wanted, all refresh
        share = torch.tensor([[0.1, 0.5, 0.9][(step + b) % 3] for b in range(B)], device="cuda").repeat_interleave(H)
        delta = torch.where(torch.rand(R, generator=g, device="cuda") < share, -1.0, 1e9).double()
        if step == 4:  # some heads without an anchor refresh whatever the gate says
            for s in (st, calls):
                s.has_anchor[::3] = 0
        both_ways(cfg, Q, K, V, delta, tau, st, ws, calls, calls_ws)
        seen.add(int(st.has_anchor.sum()))
    assert seen == {R}
