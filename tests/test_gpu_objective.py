"""The objective (Eq. 7) where the scale of its fp16 operand takes another branch, against the oracle.

The tolerance is the objective's 1e-3: both factors of every product carry one fp16 rounding of at most 2^-12, so 2^-11 =
4.9e-4 where all errors align.
"""
import numpy as np
import pytest
import torch

from oracle import gq_oracle as orc
from paper_2505_07004_b200 import api as libgq

pytestmark = pytest.mark.gpu

L_RTOL = 1e-3


@pytest.fixture(scope="module")
def dev():
    assert torch.cuda.is_available()
    torch.cuda.set_device(0)
    return torch.device("cuda:0")


def problem(d_in, d_out, g):
    rng = np.random.default_rng(d_in + 3 * d_out + g)
    X = rng.standard_normal((64, d_in)) * np.exp(rng.standard_normal(d_in))
    H = np.stack([(X * rng.random((64, 1))).T @ X for _ in range(g)]).astype(np.float32)
    H = (H + H.transpose(0, 2, 1)) / 2
    W = (0.02 * rng.standard_normal((d_out, d_in))).astype(np.float32)
    return H, W, rng


def run(dev, W, W_hat, H):
    """Two calls on a scratch full of ones: nothing in it is read before it is written, the order of every sum is fixed."""
    ws = libgq.alloc_workspace(libgq.gq_objective_workspace_bytes(H.shape[1], W.shape[0], H.shape[0]), dev)
    ws.fill_(0xFF)
    args = [torch.from_numpy(a).to(dev) for a in (W, W_hat, H)]
    first, second = (libgq.gq_objective(*args, ws).cpu().numpy() for _ in range(2))
    libgq.gq_check()
    assert np.array_equal(first, second, equal_nan=True)
    return first


def check(loss, ref):
    assert np.all(np.abs(loss - ref) <= L_RTOL * np.abs(ref)), "relative error %s" % (np.abs(loss - ref) / np.abs(ref))


# Factors around the room that the guess of the scale leaves (the sample reaches 1.4: 2 is inside, 8 is not), and far past it
@pytest.mark.parametrize("factor", [2.0, 4.0, 8.0, 16.0, 32.0, 1e6])
@pytest.mark.parametrize("at", [0, 5, -1])
def test_scale_of_outliers(dev, factor, at):
    d_in, d_out, g = 264, 1024, 2
    H, W, rng = problem(d_in, d_out, g)
    delta = (rng.integers(0, 2, W.shape) * 2 - 1) * 0.001 * (1 + 0.4 * rng.random(W.shape))
    delta.reshape(-1)[at] = 0.001 * factor
    W_hat = (W + delta).astype(np.float32)
    check(run(dev, W, W_hat, H), orc.objective(W, W_hat, H, impl="numpy"))


def test_scale_of_an_outlier_row(dev):
    """A row 300 times as wide as the others (every value of it overflows with the guessed scale, a few others are lowered into
    the subnormal range), in a layer that the second preparation kernel goes over twice."""
    d_in, d_out, g = 2312, 2320, 1
    H, W, rng = problem(d_in, d_out, g)
    delta = 0.001 * rng.standard_normal(W.shape)
    delta[1234] *= 300
    W_hat = (W + delta).astype(np.float32)
    check(run(dev, W, W_hat, H), orc.objective(W, W_hat, H, impl="numpy"))


@pytest.mark.parametrize("at", [(5, 3), (60000, 40), (120007, 71)])
def test_scale_where_blocks_share_a_byte(dev, at):
    """Few features and many channels: the scratch has no room for as many maxima as the layer has blocks, so that a block goes
    over several pieces.  The largest difference stands in a first piece, in a further one, and in the last, a partial one."""
    d_in, d_out, g = 72, 120008, 1
    H, W, rng = problem(d_in, d_out, g)
    delta = 0.001 * rng.random(W.shape)
    delta[at] = 1.0
    W_hat = (W + delta).astype(np.float32)
    check(run(dev, W, W_hat, H), orc.objective(W, W_hat, H, impl="numpy"))


def test_scale_of_a_single_difference(dev):
    """Every sample is zero; magnitudes from the smallest that the scale reaches to large ones."""
    d_in, d_out, g = 128, 4096, 1
    H, W, _ = problem(d_in, d_out, g)
    W[:] = 0
    for mag in (1e-25, 1e-6, 1.0, 1e15):
        W_hat = W.copy()
        W_hat[1234, 77] = mag
        loss = run(dev, W, W_hat, H)
        ref = float(np.float32(mag)) ** 2 * float(H[0, 77, 77])
        assert abs(loss[0] - ref) <= L_RTOL * ref and loss[1] == loss[0]
    assert not run(dev, W, W.copy(), H).any()


# The first weight always belongs to the sample that the scale is guessed from; (700, 100) does not, (1023, 263) is the last
@pytest.mark.parametrize("at", [(0, 0), (700, 100), (1023, 263)])
@pytest.mark.parametrize("bad", [np.inf, -np.inf, np.nan])
def test_differences_that_are_not_finite(dev, bad, at):
    """An infinite or undefined difference gives a loss that is not finite, for its group only; the other group's loss is what
    it is without it."""
    d_in, d_out, g = 264, 1024, 2
    H, W, rng = problem(d_in, d_out, g)
    W_hat = (W + 0.003 * rng.standard_normal(W.shape)).astype(np.float32)
    ref = orc.objective(W, W_hat, H, impl="numpy")
    W_hat[at] = bad
    loss = run(dev, W, W_hat, H)
    hit = at[0] // (d_out // g)
    assert not np.isfinite(loss[hit]) and not np.isfinite(loss[2])
    check(loss[1 - hit], ref[1 - hit])


def test_differences_that_are_all_infinite(dev):
    """No finite difference in one group, zeros in the other."""
    d_in, d_out, g = 64, 256, 2
    H, W, _ = problem(d_in, d_out, g)
    W_hat = W.copy()
    W_hat[:128] = np.inf
    loss = run(dev, W, W_hat, H)
    assert not np.isfinite(loss[0]) and loss[1] == 0.0 and not np.isfinite(loss[2])


@pytest.mark.parametrize("mantissa", [65503.0, 65504.0, 65519.9, 65520.0, 65535.0, 65536.0])
def test_scale_where_fp16_ends(dev, mantissa):
    """The largest difference lands, with the guessed scale, on either side of what fp16 can hold."""
    d_in, d_out, g = 64, 1024, 1
    H, W, _ = problem(d_in, d_out, g)
    W[:] = 0
    delta = np.full(W.shape, 16384.0 / 65536.0, dtype=np.float32)     # every sample: 2^14 with the guessed scale
    delta[5, 7] = mantissa / 65536.0
    check(run(dev, W, delta, H), orc.objective(W, delta, H, impl="numpy"))


# The last one rounds up to 2^7 in fp16
@pytest.mark.parametrize("outlier", [1.0, 3.0, 100.0, 127.99])
def test_small_group_keeps_its_bits(dev, outlier):
    """Differences 2^-28 of the layer's largest keep 11 significant bits, wherever the largest stands.

    All of the group's are equal, so every rounding error has the same sign: 2^-28 (1 + 2^-10) of the largest's power of two is
    2^-14 (1 + 2^-10) or more in fp16, exact; half of that has a bit less there, loses the 2^-10 and gives a loss 2^-9 = 1.95e-3
    too small.
    """
    d_in, d_out, g = 64, 1024, 2
    H, W, _ = problem(d_in, d_out, g)
    H = np.abs(H)
    W[:] = 0
    delta = np.full(W.shape, 1.0, dtype=np.float32)
    delta[5, 7] = outlier                                              # not in the sample
    delta[d_out // 2:] = 2.0 ** -28 * 2.0 ** np.floor(np.log2(outlier)) * (1 + 2.0 ** -10)
    check(run(dev, W, delta, H), orc.objective(W, delta, H, impl="numpy"))
