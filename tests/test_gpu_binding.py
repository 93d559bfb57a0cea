"""The binding's short way to an entry point (all tensors on the current device, no stream given) and the others."""
import pytest
import torch

from paper_2505_07004_b200 import api as libgq

pytestmark = pytest.mark.gpu


def test_stream_given_and_current_stream_agree():
    dev = torch.device("cuda", torch.cuda.current_device())
    grad = torch.randn(64, 128, device=dev).to(torch.bfloat16)
    expect = grad.float().square().view(64, 2, 64).mean(2).T
    side = torch.cuda.Stream(dev)
    side.wait_stream(torch.cuda.current_stream(dev))
    given = libgq.gq_saliency(grad, 2, stream=side)
    with torch.cuda.stream(side):
        current = libgq.gq_saliency(grad, 2)
    side.synchronize()
    plain = libgq.gq_saliency(grad, 2)
    for s in (given, current, plain):
        assert torch.allclose(s, expect, rtol=1e-5)      # sums of 64 squares in fp32: 64 * 2^-24


def test_tensors_that_are_not_all_on_the_device_are_refused():
    dev = torch.device("cuda", torch.cuda.current_device())
    X, s = torch.zeros(8, 64, dtype=torch.bfloat16, device=dev), torch.zeros(1, 8, device=dev)
    H, ws = torch.zeros(1, 64, 64, device=dev), torch.zeros(4096, dtype=torch.uint8)
    with pytest.raises(ValueError, match="workspace must be a CUDA tensor"):
        libgq.gq_hessian_accumulate(X, s, H, ws)
    with pytest.raises(libgq.GQError):                   # a status of the entry point: scratch too small
        libgq.gq_hessian_accumulate(X, s, H, ws[:8].to(dev))
