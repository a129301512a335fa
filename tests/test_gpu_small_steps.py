"""Small layer-steps, whose drift, decision and masks come from one kernel: block counts at the edges of its tiles of eight
rows and of its per-lane layouts, and shapes on both sides of the rule that picks it."""
import numpy as np
import pytest
import torch

from paper_2605_14513_b200 import inputs

from parity import Pair, check_decisions, check_masks, to_np

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nb,H,B,block", [(1, 1, 1, 64), (7, 3, 1, 128), (8, 2, 2, 64), (9, 48, 1, 64), (40, 49, 1, 64), (63, 5, 1, 64),
                                          (64, 37, 1, 64), (64, 38, 1, 64), (65, 9, 1, 64), (128, 3, 3, 128), (128, 10, 1, 64), (129, 2, 1, 64)])
def test_decision_and_masks_of_small_steps(oracle, nb, H, B, block):
    from paper_2605_14513_b200 import heart

    rs = np.random.RandomState(nb + H)
    wl = inputs.small_workload(H=H, grid=(1, 1, block * nb - 5), block=block, seed=nb, B=B, tau=rs.uniform(0.3, 0.97, B * H), pos_scale=1.0,
                               eps=np.where(np.arange(B * H) % 2 == 0, 0.003, 0.3))
    p = Pair(wl, heart, oracle)
    calls, ws = heart.State(p.cfg), heart.new_workspace(p.cfg)  # the same by separate calls
    for step in range(3):
        O, _, drift, refresh = p.gpu_step()
        d, f = torch.empty(wl.R, dtype=torch.float64, device="cuda"), torch.empty(wl.R, dtype=torch.uint8, device="cuda")
        heart.heart_drift(p.cfg, p.Q, p.K, p.delta, calls, ws, drift_out=d, refresh_out=f)
        heart.heart_predict_mask(p.cfg, p.Q, p.K, p.tau, calls, ws, refresh=f, means_valid=True)
        assert heart.heart_get_status(ws) == 0
        assert np.array_equal(to_np(d), drift) and np.array_equal(to_np(f), refresh)
        for a, b in zip(p.gst.tensors(), calls.tensors()):
            assert torch.equal(a, b)
        _, _, drift_o, refresh_o = p.oracle_step(want_O=False)
        assert check_decisions(drift, refresh, drift_o, refresh_o, wl.delta) == 0
        check_masks(p.gst, p.ost, range(wl.R), wl.tau, p.probs_row)
        p.advance()


def both_ways(cfg, Q, K, V, delta, tau, st, ws, calls, calls_ws):
    """One heart_step, and the same by separate calls on a state and a workspace of their own; the launches of the step."""
    from paper_2605_14513_b200 import heart

    R = cfg.B * cfg.H
    O, (d0, d1), (f0, f1) = torch.empty_like(Q), torch.empty((2, R), dtype=torch.float64, device="cuda"), torch.empty((2, R), dtype=torch.uint8, device="cuda")
    heart.heart_step(cfg, Q, K, V, delta, tau, st, O, ws, drift_out=d0, refresh_out=f0)
    launches = heart.heart_last_launch_count()
    heart.heart_drift(cfg, Q, K, delta, calls, calls_ws, drift_out=d1, refresh_out=f1)
    heart.heart_predict_mask(cfg, Q, K, tau, calls, calls_ws, refresh=f1, means_valid=True)
    assert heart.heart_get_status(ws) == 0 and heart.heart_get_status(calls_ws) == 0
    assert torch.equal(d0, d1) and torch.equal(f0, f1)
    for a, b in zip(st.tensors(), calls.tensors()):
        assert torch.equal(a, b)
    return launches


def random_step(g, B, H, N):
    Q, K, V = (torch.randn((B, H, N, 128), generator=g, device="cuda").to(torch.bfloat16) for _ in range(3))
    # about half of the heads refresh
    return Q, K, V, torch.where(torch.rand(B * H, generator=g, device="cuda") < 0.5, -1.0, 1e9).double()


# launches between the block sums and the attention: one kernel, the decision and the rows, or the three of larger steps
ONE, DECISION_APART, APART = 1, 2, 3


@pytest.mark.parametrize("nb,H,B,block,gate,between", [
    (32, 2, 1, 64, False, ONE), (32, 2, 1, 64, True, DECISION_APART), (40, 3, 1, 64, False, ONE), (41, 3, 1, 64, False, DECISION_APART),
    (8, 37, 1, 64, False, ONE), (8, 38, 1, 64, False, DECISION_APART), (1, 48, 1, 128, False, ONE), (1, 49, 1, 128, False, DECISION_APART),
    (8, 9, 2, 128, False, ONE), (8, 19, 1, 128, False, DECISION_APART), (24, 6, 2, 64, False, ONE), (39, 12, 2, 64, True, DECISION_APART),
    (64, 37, 1, 64, True, DECISION_APART), (64, 38, 1, 64, False, APART), (128, 9, 1, 128, False, DECISION_APART), (128, 10, 1, 128, False, APART),
    (129, 1, 1, 64, False, APART),
])
def test_which_kernels(nb, H, B, block, gate, between):
    """Both sides of the rules that pick the kernels; all the same bits."""
    from paper_2605_14513_b200 import heart

    N = nb * block - 5
    g = torch.Generator("cuda").manual_seed(nb * H)
    cfg = heart.make_config(B, H, N, block, gate_lo=0.4 if gate else 0.0, gate_hi=0.6 if gate else 1.0)
    st, calls, ws, calls_ws = heart.State(cfg), heart.State(cfg), heart.new_workspace(cfg), heart.new_workspace(cfg)
    tau = torch.linspace(0.5, 0.95, B * H, dtype=torch.float64, device="cuda")
    attention = 1 if B * H * ((N + 127) // 128) <= 148 else 3
    for step in range(3):
        assert both_ways(cfg, *random_step(g, B, H, N), tau, st, ws, calls, calls_ws) == 1 + between + attention


def test_steps_of_several_shapes_on_one_workspace():
    """The tickets of the heads are back at zero after every step, whichever kernel took them."""
    from paper_2605_14513_b200 import heart

    g = torch.Generator("cuda").manual_seed(0)
    shapes = [(1, 2, 2043, 64), (1, 37, 500, 64), (2, 3, 1000, 128), (1, 12, 2500, 64)]
    cfgs = [heart.make_config(*s) for s in shapes]
    ws = heart.new_workspace(max(cfgs, key=heart.workspace_bytes))
    own = [(heart.State(c), heart.State(c), heart.new_workspace(c)) for c in cfgs]
    for step in range(3):
        for (B, H, N, block), cfg, (st, calls, calls_ws) in zip(shapes, cfgs, own):
            tau = torch.full((B * H,), 0.8, dtype=torch.float64, device="cuda")
            both_ways(cfg, *random_step(g, B, H, N), tau, st, ws, calls, calls_ws)
