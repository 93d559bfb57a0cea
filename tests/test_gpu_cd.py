"""GPU parity of gq_cd_cycles (cyclic coordinate descent with fixed codebooks, Eq. 10 / Algorithm 4) against
the CPU fp64 oracle.

Rounding decisions are integers decided by floating point, and the two sides sum in different precisions and
orders, so a decision can legitimately differ where the rounding target lies (numerically) on the midpoint
between two codebook values; from that coordinate on the channel follows a different, equally valid descent
path.  The tests therefore require
  * identical codes for every channel except where the oracle itself certifies such a near-tie at the FIRST
    coordinate where the codes differ (one cycle: the state before that coordinate is identical on both sides);
  * for every channel, whatever path it took: W_hat[j][i] == codebook[j][Q[j][i]] exactly, and the channel's
    objective (fp64, Eq. 7 restricted to the channel) does not exceed its starting value;
  * group totals of the objective within 1e-3 of the oracle's.
"""
import numpy as np
import pytest
import torch

from oracle import cd_oracle as cdo
from paper_2505_07004_b200 import api as libgq

pytestmark = pytest.mark.gpu

TIE_RTOL = 2e-4          # |distance to GPU's value - distance to oracle's value| <= TIE_RTOL * magnitude of the sum


@pytest.fixture(scope="module")
def dev():
    assert torch.cuda.is_available()
    torch.cuda.set_device(0)
    return torch.device("cuda:0")


def make_problem(seed, d_in, d_out, g, m, n=None, dead=()):
    rng = np.random.default_rng(seed)
    n = n or 2 * d_in
    X = rng.standard_normal((n, d_in)) * np.exp(0.7 * rng.standard_normal(d_in))
    X[:, list(dead)] = 0.0
    H = np.stack([(X * (rng.random((n, 1)) * np.exp(rng.standard_normal((n, 1))))).T @ X for _ in range(g)])
    H = ((H + H.transpose(0, 2, 1)) / 2).astype(np.float32)
    W = (0.02 * rng.standard_normal((d_out, d_in))).astype(np.float32)
    lo, hi = W.min(1, keepdims=True), W.max(1, keepdims=True)
    grid = lo + (hi - lo) * (np.arange(m)[None, :] + 0.5 * rng.random((d_out, m))) / m       # non-uniform levels
    cb = grid.astype(np.float32)
    W0, _ = cdo.round_to_codebook(W, cb)
    return W, W0.astype(np.float32), cb, H


def run_gpu(dev, W, W0, cb, H, cycles):
    Wd, Whd = torch.from_numpy(W).to(dev), torch.from_numpy(W0.copy()).to(dev)
    cbd, Hd = torch.from_numpy(cb).to(dev), torch.from_numpy(H).to(dev)
    ws = libgq.alloc_workspace(libgq.gq_cd_workspace_bytes(W.shape[1], W.shape[0], H.shape[0]), dev)
    What, Q = libgq.gq_cd_cycles(Wd, Whd, cbd, Hd, cycles, ws)
    libgq.gq_check()
    return What.cpu().numpy(), Q.cpu().numpy().astype(np.int32)


def per_channel_objective(W, What, H):
    mk = W.shape[0] // H.shape[0]
    return np.array([cdo.channel_objective(What[j].astype(np.float64) - W[j], H[j // mk].astype(np.float64))
                     for j in range(W.shape[0])])


def check_against_oracle(W, W0, cb, H, What_g, Q_g, cycles, certify_ties):
    d_out, d_in = W.shape
    mk = d_out // H.shape[0]
    What_o, Q_o = cdo.cd(W, W0, cb, H, cycles, 128)
    # feasibility and descent for every channel
    assert Q_g.min() >= 0 and Q_g.max() < cb.shape[1]
    assert np.array_equal(What_g, np.take_along_axis(cb, Q_g, axis=1)), "W_hat must be codebook[Q] exactly"
    f0, fg, fo = (per_channel_objective(W, x, H) for x in (W0, What_g, What_o))
    assert np.all(fg <= f0 * (1 + 1e-6) + 1e-30), "a channel's objective went up"
    diff = np.nonzero((Q_g != Q_o).any(axis=1))[0]
    if certify_ties:
        for j in diff:
            i = int(np.nonzero(Q_g[j] != Q_o[j])[0][0])          # first coordinate in processing order
            state = W0[j].astype(np.float64).copy()
            state[:i] = What_o[j, :i]                            # identical on both sides before i
            t, mag = cdo.coordinate_target(W[j], state, H[j // mk], i)
            da, db = abs(t - float(cb[j, Q_g[j, i]])), abs(t - float(cb[j, Q_o[j, i]]))
            assert abs(da - db) <= TIE_RTOL * mag, \
                "channel %d coordinate %d: GPU took level %d, oracle %d, target %.9g is no near-tie (%.3e vs %.3e, scale %.3e)" \
                % (j, i, Q_g[j, i], Q_o[j, i], t, da, db, mag)
    assert len(diff) <= max(2, 0.05 * d_out), "%d of %d channels differ from the oracle" % (len(diff), d_out)
    tg, to = fg.reshape(-1, mk).sum(1), fo.reshape(-1, mk).sum(1)
    assert np.all(np.abs(tg - to) <= 1e-3 * to), "group objectives %s vs oracle %s" % (tg, to)
    return len(diff)


@pytest.mark.parametrize("seed,d_in,d_out,g,m", [
    (0, 128, 64, 2, 4),         # one block, no panel product
    (1, 328, 96, 3, 8),         # two blocks, the second ragged (72 coordinates); 32 channels per group
    (2, 520, 48, 2, 16),        # three blocks; 24 channels per group (a half filled slice of 16 channels)
    (3, 1032, 256, 1, 2),       # five blocks, one group, binary codebooks
    (4, 768, 1024, 2, 4),       # two channel tiles of 256 per group
])
def test_cd_one_cycle_matches_oracle(dev, seed, d_in, d_out, g, m):
    W, W0, cb, H = make_problem(seed, d_in, d_out, g, m)
    What_g, Q_g = run_gpu(dev, W, W0, cb, H, 1)
    check_against_oracle(W, W0, cb, H, What_g, Q_g, 1, certify_ties=True)


def test_cd_several_cycles_and_dead_feature(dev):
    W, W0, cb, H = make_problem(7, 600, 128, 2, 8, dead=(5, 300))
    assert H[0, 5, 5] == 0.0 and H[1, 300, 300] == 0.0
    What_g, Q_g = run_gpu(dev, W, W0, cb, H, 3)
    check_against_oracle(W, W0, cb, H, What_g, Q_g, 3, certify_ties=False)
    # dead features are rounded to the value nearest to W
    val, q = cdo.round_to_codebook(W[:, [5, 300]], cb)
    assert np.array_equal(Q_g[:, [5, 300]], q)
    # a second call continues from where the first stopped: 2 + 1 cycles == 3 cycles
    W2, Q2 = run_gpu(dev, W, W0, cb, H, 2)
    W3, Q3 = run_gpu(dev, W, W2, cb, H, 1)
    assert np.array_equal(Q3, Q_g) and np.array_equal(W3, What_g)


def test_cd_llama_shaped_group(dev):
    """d_in 2048, 2 groups of 512 channels, 4-bit codebooks: several panel pieces per tile, two cycles."""
    W, W0, cb, H = make_problem(11, 2048, 1024, 2, 16, n=3000)
    What_g, Q_g = run_gpu(dev, W, W0, cb, H, 1)
    n_diff = check_against_oracle(W, W0, cb, H, What_g, Q_g, 1, certify_ties=True)
    print("channels on a different (near-tie) path: %d of %d" % (n_diff, W.shape[0]))


@pytest.mark.parametrize("seed,d_in,d_out,g,m", [
    (20, 296, 88, 1, 3),        # five channel slices of 16 and one of 8; second block of 40 coordinates: a band and a quarter
    (21, 512, 40, 1, 5),        # whole blocks
    (22, 264, 72, 3, 13),       # second block of 8 coordinates
])
def test_cd_block_edges(dev, seed, d_in, d_out, g, m):
    """Level counts between the block kernel's 4, 8 and 16, in no order and with a level given twice (the codes name the
    first of the two), ragged bands and channel slices."""
    W, W0, cb, H = make_problem(seed, d_in, d_out, g, m)
    cb = cb[:, np.random.default_rng(seed).permutation(m)].copy()
    cb[:, m - 1] = cb[:, 0]
    W0 = cdo.round_to_codebook(W, cb)[0].astype(np.float32)
    What_g, Q_g = run_gpu(dev, W, W0, cb, H, 1)
    check_against_oracle(W, W0, cb, H, What_g, Q_g, 1, certify_ties=True)
    assert Q_g.max() < m - 1


# narrow layers (16 channels per CTA); and one of 32 per CTA, the last slice of a group with 8, in one block of coordinates
@pytest.mark.parametrize("m,d_in,d_out,g", [(4, 264, 64, 2), (8, 264, 64, 2), (13, 264, 64, 2), (16, 264, 64, 2), (3, 256, 2424, 3),
                                            (8, 256, 2424, 3), (16, 256, 2424, 3)])
def test_cd_levels_that_are_no_numbers(dev, m, d_in, d_out, g):
    """A NaN level is never chosen while its channel has a number: the channel ends where it ends with that level far
    away.  A channel of NaN only, or with a NaN in W, still gets codes below m, and its neighbours (four channels share a
    word of codes) the bits they get without it."""
    W, W0, cb, H = make_problem(40 + m, d_in, d_out, g, m)
    far = cb.copy()
    far[3, m // 2] = far[9, 0] = far[50, m - 1] = 1e30
    What_f, Q_f = run_gpu(dev, W, W0, far, H, 2)
    W_n, cb_n = W.copy(), far.copy()
    cb_n[far == 1e30] = np.nan
    cb_n[5] = np.nan
    W_n[22, 100] = np.nan
    What_n, Q_n = run_gpu(dev, W_n, W0, cb_n, H, 2)
    assert Q_n.max() < m
    assert np.array_equal(What_n, np.take_along_axis(cb_n, Q_n, axis=1), equal_nan=True)
    assert (Q_n[5] == 0).all()
    rest = [j for j in range(d_out) if j not in (5, 22)]
    assert np.array_equal(Q_n[rest], Q_f[rest]) and np.array_equal(What_n[rest], What_f[rest])


def test_cd_more_panel_tiles_than_pairs(dev):
    """80 groups of 8 channels: 80 panel units on at most 74 CTA pairs, some pairs take two and add their tiles to P
    without the staging ring; two ragged panels."""
    W, W0, cb, H = make_problem(50, 520, 640, 80, 4, n=600)
    What_g, Q_g = run_gpu(dev, W, W0, cb, H, 1)
    check_against_oracle(W, W0, cb, H, What_g, Q_g, 1, certify_ties=True)


@pytest.mark.parametrize("value", [np.nan, np.inf])
def test_cd_does_not_look_at_the_first_start_value(dev, value):
    """Coordinate 0 is set before anything reads W_hat[:, 0]: whatever stands there, the result is the same bits."""
    W, W0, cb, H = make_problem(60, 264, 40, 1, 4)
    W_any = W0.copy()
    W_any[:, 0] = value
    want, got = run_gpu(dev, W, W0, cb, H, 1), run_gpu(dev, W, W_any, cb, H, 1)
    assert np.array_equal(got[0], want[0]) and np.array_equal(got[1], want[1])


def test_cd_errors_and_zero_cycles(dev):
    W, W0, cb, H = make_problem(3, 64, 16, 1, 4)
    Wd, Whd = torch.from_numpy(W).to(dev), torch.from_numpy(W0.copy()).to(dev)
    cbd, Hd = torch.from_numpy(cb).to(dev), torch.from_numpy(H).to(dev)
    ws = libgq.alloc_workspace(libgq.gq_cd_workspace_bytes(64, 16, 1), dev)
    What, Q = libgq.gq_cd_cycles(Wd, Whd, cbd, Hd, 0, ws)
    libgq.gq_check()
    assert np.array_equal(What.cpu().numpy(), W0)
    with pytest.raises(libgq.GQError) as e:
        libgq.gq_cd_cycles(Wd, Whd, cbd, Hd, 1, ws[:1024])
    assert "GQ_ERR_WORKSPACE" in str(e.value)
    big = torch.zeros((16, 17), device=dev)
    with pytest.raises(libgq.GQError) as e:
        libgq.gq_cd_cycles(Wd, Whd, big, Hd, 1, ws)
    assert "GQ_ERR_UNSUPPORTED_SHAPE" in str(e.value)
    assert libgq.gq_cd_workspace_bytes(60, 16, 1) == 0
