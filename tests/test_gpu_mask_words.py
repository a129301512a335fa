"""Rows of every number of mask words: the kernels of the top-p rows and of the antidiagonal importances have an instance for each even
number of them, and the rows of a CTA and the registers of a thread go by it."""
import numpy as np
import pytest
import torch

from paper_2605_14513_b200 import inputs

from parity import Pair, check_masks

pytestmark = pytest.mark.gpu


def pair(oracle, nb, H, block, flags=0):
    from paper_2605_14513_b200 import heart

    rs = np.random.RandomState(nb + block)
    wl = inputs.small_workload(H=H, grid=(1, 1, block * nb - 5), block=block, seed=nb, tau=rs.uniform(0.5, 0.97, H), pos_scale=1.5)
    p = Pair(wl, heart, oracle)
    p.cfg.flags |= flags
    return heart, wl, p


@pytest.mark.parametrize("words", range(1, 33))
def test_top_p_rows(oracle, words):
    for nb in {32 * words - 31, 32 * words}:  # one block in the last word, and a whole one
        heart, wl, p = pair(oracle, nb, 1, 64)
        heart.heart_predict_mask(p.cfg, p.Q, p.K, p.tau, p.gst, p.ws)
        assert heart.heart_get_status(p.ws) == 0
        oracle.predict_mask(p.Qb, p.Kb, wl.block, wl.tau, p.ost)
        assert check_masks(p.gst, p.ost, range(wl.R), wl.tau, p.probs_row) == 0


@pytest.mark.parametrize("block,nb", [(64, 3), (64, 64), (64, 65), (64, 129), (64, 200), (128, 2), (128, 65), (128, 97), (128, 161)])
def test_antidiagonal_rows(oracle, block, nb):
    from paper_2605_14513_b200 import heart as h

    heart, wl, p = pair(oracle, nb, 2 if nb < 100 else 1, block, h.ESTIMATOR_ANTIDIAG)
    ws = heart.new_workspace(p.cfg)
    heart.heart_predict_mask(p.cfg, p.Q, p.K, p.tau, p.gst, ws)
    assert heart.heart_get_status(ws) == 0
    oracle.predict_mask_antidiag(p.Qb, p.Kb, wl.block, wl.tau, p.ost)
    # importances from bf16 products with fp32 sums: a row may cut elsewhere within the bands of check_masks
    assert check_masks(p.gst, p.ost, range(wl.R), wl.tau, lambda r, I: oracle.antidiag_probs_row(p.Qb, p.Kb, block, r, I)) <= 2
