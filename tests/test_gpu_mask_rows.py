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


@pytest.mark.parametrize("base,step", [(0.0, 2.0 ** -57), (0.0, 2.0 ** -54), (0.75, 2.0 ** -53), (0.75, 2.0 ** -49)])
@pytest.mark.parametrize("nb", [4, 40, 600])
def test_scores_a_rounding_apart(oracle, base, step, nb):
    """Scores base + {0 .. 3} * step: where exp(score - max) is the same double the lowest index comes first, although
    the fp32 values of score - max differ; where it is not, the larger score does."""
    from paper_2605_14513_b200 import heart

    rs = np.random.RandomState(nb)
    times = rs.randint(0, 4, nb)
    times[:4] = [0, 1, 2, 0]
    N = 64 * nb
    K = torch.zeros((1, 1, nb, 64, 128))
    K[..., 0] = base
    K[..., 1] = torch.from_numpy(times * step).float()[None, None, :, None]
    K = K.view(1, 1, N, 128).to(torch.bfloat16).cuda()
    Q = torch.zeros((1, 1, N, 128))
    Q[..., :2] = 1.0
    Q = Q.to(torch.bfloat16).cuda()
    cfg = heart.make_config(1, 1, N, 64, scale=1.0)
    # (weights equal to 1e-14: cuts lie near k / nb, where a mass is within rounding of tau; these stay 2e-4 away)
    for tau in (0.3137, 0.4231, 0.7139, 0.9173):
        st, ost, ws = heart.State(cfg), oracle.State(1, 1, N, 128, 64), heart.new_workspace(cfg)
        heart.heart_predict_mask(cfg, Q, K, torch.tensor([tau], dtype=torch.float64, device="cuda"), st, ws)
        oracle.predict_mask(inputs.bits(Q), inputs.bits(K), 64, np.array([tau]), ost, scale=1.0)
        assert np.array_equal(st.kv_cnt.cpu().numpy(), ost.kv_cnt)
        assert np.array_equal(st.mask_bits.cpu().numpy().view(np.uint32), ost.mask_bits)


@pytest.mark.parametrize("nb", [3, 64, 65, 130, 700])
def test_rows_of_equal_scores(oracle, nb):
    """All blocks equal, all but one, half of them, and equal ones below the cut: more than 64 candidates that no
    threshold parts."""
    from paper_2605_14513_b200 import heart

    N = 64 * nb
    rs = np.random.RandomState(nb)
    score = np.zeros((4, nb))
    score[1, nb // 2] = 3.0
    score[2, rs.permutation(nb)[: nb // 2]] = 1.5
    score[3] = np.where(np.arange(nb) % 3 == 0, -2.0, rs.uniform(-1, 1, nb))
    K = torch.zeros((1, 4, nb, 64, 128))
    K[..., 0] = torch.from_numpy(score).float()[None, :, :, None]
    K = K.view(1, 4, N, 128).to(torch.bfloat16).cuda()
    Q = torch.zeros((1, 4, N, 128))
    Q[..., 0] = 1.0
    Q = Q.to(torch.bfloat16).cuda()
    cfg = heart.make_config(1, 4, N, 64, scale=1.0)
    for tau in (0.0137, 0.3137, 0.7139, 0.9773):  # (not within rounding of k / nb, where the mass of equal blocks is)
        tau = np.full(4, tau)
        st, ost, ws = heart.State(cfg), oracle.State(1, 4, N, 128, 64), heart.new_workspace(cfg)
        heart.heart_predict_mask(cfg, Q, K, torch.from_numpy(tau).cuda(), st, ws)
        oracle.predict_mask(inputs.bits(Q), inputs.bits(K), 64, tau, ost, scale=1.0)
        assert np.array_equal(st.kv_cnt.cpu().numpy(), ost.kv_cnt)
        assert np.array_equal(st.mask_bits.cpu().numpy().view(np.uint32), ost.mask_bits)
