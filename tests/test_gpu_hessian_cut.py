"""Hessian launches whose last round of units is cut along the tokens: evenly per unit, or across units."""
import numpy as np
import pytest
import torch

from oracle import gq_oracle as orc
from paper_2505_07004_b200 import api as libgq
from paper_2505_07004_b200 import synth
from test_gpu_parity import check_H, dev, gpu_hessian  # noqa: F401

pytestmark = pytest.mark.gpu


# one unit and one k-step; one unit of many k-steps; two units; as many k-steps as the smallest piece and one more; a last piece
# that is one k-step longer; odd groups; more units than half of the pairs; whole rounds and a remainder that is cut across units
@pytest.mark.parametrize("d_in,n,g", [(256, 40, 1), (256, 2048, 1), (256, 1100, 4), (512, 128, 2), (512, 129, 2), (264, 1000, 3),
                                      (1536, 200, 1), (1032, 330, 3), (1288, 1500, 8)])
def test_cut_last_round(dev, d_in, n, g):  # noqa: F811
    gen = torch.Generator(device=dev).manual_seed(d_in + n + g)
    X = (torch.randn(n, d_in, generator=gen, device=dev) * torch.exp(torch.randn(d_in, generator=gen, device=dev))).to(torch.bfloat16)
    s = torch.rand(g, n, generator=gen, device=dev) + 0.1
    H = gpu_hessian([X, X], [s, s], d_in, g, dev)                     # twice: pieces add to what is there
    check_H(H, 2 * orc.hessian(synth.bf16_bits(X), s.cpu().numpy().astype(np.float64)))
