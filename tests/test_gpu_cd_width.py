"""Coordinate descent on both sides of the layer width from which a CTA of the block kernel takes 32 channels instead of 16."""
import numpy as np
import pytest
import torch

from oracle import cd_oracle as cdo
from test_gpu_cd import check_against_oracle, dev, make_problem, run_gpu  # noqa: F401

pytestmark = pytest.mark.gpu


def narrowest_wide(dev):
    """One channel row of 8 more than the SMs can take 16 at a time."""
    return 16 * torch.cuda.get_device_properties(dev).multi_processor_count + 8


# one block of coordinates (no panel product, so every sum has a fixed order), whole and ragged
@pytest.mark.parametrize("m", [3, 8, 16])
@pytest.mark.parametrize("d_in", [256, 72])
def test_sixteen_and_thirty_two_channels_agree(dev, d_in, m):
    wide = narrowest_wide(dev)
    W, W0, cb, H = make_problem(11 + m, d_in, wide, 1, m)
    What_w, Q_w = run_gpu(dev, W, W0, cb, H, 2)
    What_n, Q_n = run_gpu(dev, W[:-8], W0[:-8], cb[:-8], H, 2)
    assert np.array_equal(Q_w[:-8], Q_n) and np.array_equal(What_w[:-8], What_n)


@pytest.mark.parametrize("m", [4, 16])
def test_thirty_two_channels_match_oracle(dev, m):
    W, W0, cb, H = make_problem(23 + m, 296, narrowest_wide(dev), 1, m)
    What_g, Q_g = run_gpu(dev, W, W0, cb, H, 1)
    check_against_oracle(W, W0, cb, H, What_g, Q_g, 1, certify_ties=True)


# Three groups of 808 channels: 32 per CTA, the last of a group's slices with 8, beside the next group's channels
@pytest.mark.parametrize("m,d_in,cycles", [(4, 296, 1), (7, 296, 1), (13, 264, 1), (16, 520, 1), (5, 520, 3), (16, 296, 2)])
def test_thirty_two_channels_in_groups(dev, m, d_in, cycles):
    """Levels in no order and one of them twice (the codes name the first), dead features, ragged blocks, one cycle and more."""
    d_out, g, dead = 2424, 3, (5, d_in - 3)
    assert g * -(-(d_out // g) // 16) > torch.cuda.get_device_properties(dev).multi_processor_count
    W, W0, cb, H = make_problem(70 + m, d_in, d_out, g, m, dead=dead)
    cb = cb[:, np.random.default_rng(m).permutation(m)].copy()
    cb[:, m - 1] = cb[:, 0]
    W0 = cdo.round_to_codebook(W, cb)[0].astype(np.float32)
    What_g, Q_g = run_gpu(dev, W, W0, cb, H, cycles)
    check_against_oracle(W, W0, cb, H, What_g, Q_g, cycles, certify_ties=cycles == 1)
    assert Q_g.max() < m - 1
    assert np.array_equal(Q_g[:, list(dead)], cdo.round_to_codebook(W[:, list(dead)], cb)[1])
