"""Hessian launches whose last round of units is cut along the tokens: evenly per unit, or across units."""
import numpy as np
import pytest
import torch

from oracle import gq_oracle as orc
from paper_2505_07004_b200 import api as libgq
from paper_2505_07004_b200 import synth
from test_gpu_parity import check_H, dev, gpu_hessian  # noqa: F401

pytestmark = pytest.mark.gpu


# (features, tokens, groups); which way a launch goes with 74 pairs, and why it stands here, is asserted in tests/test_schedule.py.
# one unit and one k-step; one unit of many k-steps; two units; as many k-steps as the smallest piece and one more; five units of
# three groups; more pieces than one per unit; most pairs with a whole unit; whole rounds, then pieces that differ by a k-step
EVENLY = [(256, 40, 1), (256, 2048, 1), (256, 1100, 4), (512, 128, 2), (512, 129, 2), (264, 1000, 3), (1536, 200, 1), (1032, 330, 3),
          (1536, 200, 4), (520, 5000, 1), (1288, 1500, 8)]
# pieces of two units for most pairs, of different lengths, ragged token counts; 26, 42 and 72 units; 70 behind a whole round
ACROSS = [(1032, 2501, 3), (1536, 2500, 4), (2048, 1100, 4), (1800, 1500, 8)]


@pytest.mark.parametrize("d_in,n,g", EVENLY + ACROSS)
def test_cut_last_round(dev, d_in, n, g):  # noqa: F811
    gen = torch.Generator(device=dev).manual_seed(d_in + n + g)
    X = (torch.randn(n, d_in, generator=gen, device=dev) * torch.exp(torch.randn(d_in, generator=gen, device=dev))).to(torch.bfloat16)
    s = torch.rand(g, n, generator=gen, device=dev) + 0.1
    H = gpu_hessian([X, X], [s, s], d_in, g, dev)                     # twice: pieces add to what is there
    check_H(H, 2 * orc.hessian(synth.bf16_bits(X), s.cpu().numpy().astype(np.float64)))


def test_saliency_ahead_of_a_cut_launch(dev):  # noqa: F811
    """26 units cut evenly over 52 pairs, whose spare warps share the next chunk's saliency between them."""
    d_in, n, g, d_out, next_n = 1032, 2048, 3, 72, 701
    gen = torch.Generator(device=dev).manual_seed(9)
    X = (torch.randn(n, d_in, generator=gen, device=dev) * torch.exp(torch.randn(d_in, generator=gen, device=dev))).to(torch.bfloat16)
    s = torch.rand(g, n, generator=gen, device=dev) + 0.1
    grad = torch.randn(next_n, d_out, generator=gen, device=dev).to(torch.bfloat16)
    H = torch.zeros(g, d_in, d_in, device=dev)
    ws, next_ws, plain_ws = (libgq.alloc_workspace(libgq.gq_hessian_workspace_bytes(n, d_in, g), dev) for _ in range(3))
    before = libgq.gq_launch_count()
    next_s = libgq.gq_hessian_accumulate_ahead(X, s, H, ws, grad, next_ws)
    assert libgq.gq_launch_count() - before == 2                      # split of s, Hessian: the saliency has no launch of its own
    plain_s = libgq.gq_saliency_prepared(grad, g, plain_ws)
    libgq.gq_hessian_finalize(H)
    libgq.gq_check()
    check_H(H, orc.hessian(synth.bf16_bits(X), s.cpu().numpy().astype(np.float64)))
    words = 8 * ((g + 1) // 2) * next_n
    assert torch.equal(next_s, plain_s) and torch.equal(next_ws[:words], plain_ws[:words])


def test_error_of_a_long_launch(dev):  # noqa: F811
    """16384 tokens of 4096 features, one group: 72 units for (at most) 74 pairs.  Accumulated in two shorter runs each, as most
    of them are where the units are cut across the pairs, H is 2.36e-4 from 64 bits; in one run of 256 k-steps each, whose
    truncated additions weigh more, 2.79e-4.  (The rest is the one bf16 rounding of every product, the same either way.)"""
    d_in, n = 4096, 16384
    syn = synth.LayerSynth(synth.LayerConfig("long", n, n, d_in, 512, (1,), "lognormal", 0.01, 20.0), dev, 2)
    X = syn.x_chunk(0)
    gen = torch.Generator(device=dev).manual_seed(7)
    s = torch.exp(2 * torch.randn(1, n, generator=gen, device=dev))
    H = gpu_hessian([X], [s], d_in, 1, dev)
    exact = (X.double() * s[0, :, None].double()).T @ X.double()
    error = float((H[0].double() - exact).norm() / exact.norm())
    assert error <= 2.55e-4, "error against 64 bits %.3e" % error
