"""The fp16 differences of the objective brought from one power of two to a smaller one in place (gq_gram_dot.cuh), compiled for
the host: wherever that is done, it gives what rounding the difference itself at the smaller scale gives."""
import os
import subprocess

import numpy as np
import pytest

from paper_2505_07004_b200 import build as gq_build

HERE = os.path.dirname(os.path.abspath(__file__))
DOWN = (1, 2, 3, 5, 10, 14, 24, 28, 29, 30, 31, 100, 200)


@pytest.fixture(scope="module")
def lowered(tmp_path_factory):
    exe = str(tmp_path_factory.mktemp("lower") / "lower")
    subprocess.check_call([gq_build._nvcc(), "-gencode", "arch=compute_100a,code=sm_100a", "-std=c++17", "-o", exe,
                           os.path.join(HERE, "delta_lower.cu")])
    out = np.frombuffer(subprocess.check_output([exe] + [str(d) for d in DOWN]), dtype=np.uint32)
    return out.reshape(len(DOWN), 65536)


@pytest.mark.parametrize("i", range(len(DOWN)))
def test_lowering_is_rounding_at_the_smaller_scale(lowered, i):
    ok, result = lowered[i] >> 16 != 0, (lowered[i] & 0xffff).astype(np.uint16).view(np.float16)
    h = np.arange(65536, dtype=np.uint16).view(np.float16)
    value = h.astype(np.float64)
    finite = np.isfinite(value)
    assert not ok[~finite].any() and ok[value == 0].all()
    want = np.zeros(65536, dtype=np.float64)
    want[finite] = np.ldexp(value[finite], -DOWN[i])
    normal = np.abs(want) >= 2.0 ** -14
    assert np.array_equal(ok[finite], (normal | (value == 0))[finite])       # the others are rounded again
    assert np.array_equal(result[ok].view(np.uint16), want[ok].astype(np.float16).view(np.uint16))
    # the ends of what rounds to h, just inside: half a unit in the last place on either side
    ulp = np.ldexp(1.0, np.maximum(np.where(value == 0, -13, np.frexp(np.where(finite, value, 0.0))[1]), -13) - 11)
    for side in (-0.49, 0.49):
        near = np.where(ok, value, 0.0) + side * ulp
        use = ok & (near.astype(np.float16) == h)
        assert use.any() and np.array_equal(np.ldexp(near[use], -DOWN[i]).astype(np.float16), result[use])
