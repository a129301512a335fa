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
