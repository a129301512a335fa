"""The band error's two ways, plane by plane in two launches and axis by axis in five, at the edges of their tiles and of the
rule between them: axes of length 1 and 2, lines that do not fill a CTA, axes with more folded samples than one
shared-memory chunk holds (more than 318) or than the shared table (1024)."""
import numpy as np
import pytest
import torch

from parity import to_np

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("shape", [(1, 1, 1, 1), (1, 2, 1, 3), (3, 1, 7, 2), (2, 4, 1, 319), (1, 400, 3, 2), (1, 2, 1030, 4), (1, 21, 60, 104)])
def test_band_error_axes(oracle, shape):
    from paper_2605_14513_b200 import heart

    g = torch.Generator("cuda").manual_seed(sum(shape))
    yd = torch.randn(shape, device="cuda", generator=g)
    ys = (yd + 0.1 * torch.randn(shape, device="cuda", generator=g)).contiguous()
    out = to_np(heart.heart_band_error(ys, yd))
    e, bands, denom = oracle.band_error(to_np(ys), to_np(yd))
    # fp64 sums of at most n terms a pass: 1e-12 of the total covers n = 1030 with a wide margin
    assert np.allclose(out[1:5], bands, rtol=1e-9, atol=1e-12 * bands.sum())
    assert np.isclose(out[5], denom, rtol=1e-12) and np.isclose(out[0], e, rtol=1e-9)


@pytest.mark.parametrize("shape", [(1, 1, 1, 4097), (5, 700, 2, 3), (1, 3, 2048, 1), (146, 1, 64, 65)])
def test_few_long_lines(oracle, shape):
    """Axes whose lines are fewer than the SMs: CTAs share their frequencies (one to 65 shares of them, uneven ones)."""
    test_band_error_axes(oracle, shape)


@pytest.mark.parametrize("shape", [(1, 1, 8, 64), (2, 3, 23, 23), (1, 5, 1, 512), (3, 2, 512, 1), (1, 4, 2, 257), (1, 2, 257, 2), (3, 96, 16, 33),
                                   (1, 97, 16, 33), (2, 2, 96, 170), (1, 3, 97, 169), (1, 1, 110, 215), (1, 1, 7, 73), (40, 1, 30, 41)])
def test_planes_in_shared_memory(oracle, shape):
    """Planes on both sides of what a CTA takes (512 points, its shared memory, 96 steps of time), axes that fill their
    tiles of eight lines and frequencies and axes that do not.  (Which way a shape takes: test_which_way.)"""
    test_band_error_axes(oracle, shape)


AXES, PLANES = 5, 2  # launches


@pytest.mark.parametrize("shape,launches", [
    # axis by axis: y axes of several chunks, beyond the shared table, of shared frequencies; some hundred CTAs a pass
    ((1, 2, 330, 80), AXES), ((1, 2, 1030, 4), AXES), ((1, 2, 2050, 16), AXES), ((1, 3, 2048, 1), AXES), ((4, 3, 120, 220), AXES),
    # planes that do not fit a CTA, at most 511 points, more than 96 steps of time
    ((1, 1, 110, 215), AXES), ((1, 1, 7, 73), AXES), ((1, 1, 8, 64), PLANES), ((1, 97, 16, 33), AXES), ((3, 96, 16, 33), PLANES),
    # one plane an SM: about a wave of them (61 to 148 CTAs)
    ((1, 30, 90, 160), AXES), ((1, 31, 90, 160), PLANES), ((2, 37, 90, 160), PLANES), ((3, 25, 90, 160), AXES), ((2, 16, 109, 201), PLANES),
    ((16, 13, 90, 160), AXES),
    # narrow planes
    ((1, 5, 1, 512), AXES), ((1, 2, 257, 2), PLANES), ((1, 4, 2, 257), AXES), ((2, 90, 16, 90), PLANES), ((37, 8, 23, 25), PLANES), ((149, 2, 23, 25), AXES), ((5, 40, 5, 107), AXES),
    ((16, 2, 160, 20), PLANES), ((15, 5, 160, 20), AXES),
    # small ones: up to 888 CTAs
    ((12, 37, 24, 24), PLANES), ((12, 38, 24, 24), AXES),
    # long chains: enough CTAs for all SMs, and for a second one on most of them
    ((4, 7, 72, 144), AXES), ((5, 15, 72, 144), PLANES), ((4, 21, 68, 104), AXES), ((4, 28, 68, 104), PLANES), ((1, 21, 60, 104), PLANES),
])
def test_which_way(oracle, shape, launches):
    from paper_2605_14513_b200 import heart

    test_band_error_axes(oracle, shape)
    assert heart.heart_last_launch_count() == launches
