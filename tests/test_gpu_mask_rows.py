"""Mask rows whose cut lies next to tau: the fp32 decision of the top-p kernel must hand them to fp64.  For
every head, tau is put 1e-9 to 1e-4 above or below a cumulative mass of one of its rows (fp64 oracle), over
block counts at the edges of the score tiles (32 and 64 blocks) and of the per-lane row layouts."""
import numpy as np
import pytest
import torch

from paper_2605_14513_b200 import inputs

from parity import Pair, check_masks

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nb,H", [(1, 2), (2, 2), (31, 8), (33, 8), (64, 8), (65, 8), (257, 4), (513, 2), (769, 1)])
def test_thresholds_next_to_a_cumulative_mass(oracle, nb, H):
    from paper_2605_14513_b200 import heart

    rs = np.random.RandomState(nb)
    wl = inputs.small_workload(H=H, grid=(1, 1, 64 * nb - 5), block=64, seed=nb, tau=np.full(H, 0.9), pos_scale=1.0)
    p = Pair(wl, heart, oracle)
    tau = np.empty(H)
    for r in range(H):
        cum = np.cumsum(np.sort(p.probs_row(r, int(rs.randint(nb))))[::-1])
        k = min(int(np.searchsorted(cum, rs.uniform(0.3, 0.97))), nb - 1)
        tau[r] = cum[k] * (1 + (-1) ** r * 10.0 ** -rs.uniform(4, 9))
    wl.tau[:] = tau
    p.tau = torch.tensor(tau, dtype=torch.float64, device="cuda")
    heart.heart_predict_mask(p.cfg, p.Q, p.K, p.tau, p.gst, p.ws)
    assert heart.heart_get_status(p.ws) == 0
    oracle.predict_mask(p.Qb, p.Kb, wl.block, tau, p.ost)
    # fp64 on both sides: cuts 1e-9 apart are told apart
    assert check_masks(p.gst, p.ost, range(H), tau, p.probs_row) == 0
