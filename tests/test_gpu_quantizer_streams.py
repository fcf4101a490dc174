"""The quantizer's streams where a warp's run of 512 columns begins, ends or is cut short, and on both sides of the zero
point (2^20) up to which codes are formed by an integer add; bit for bit against the oracle."""
import numpy as np
import pytest
import torch

import oracle as O
from paper_2407_08296_b200 import binding as B

from parity_utils import f32_to_device, from_device_q

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("bits", [2, 4, 8])
@pytest.mark.parametrize("cols", [3, 129, 511, 513, 769, 1025])
def test_runs_and_zero_points(bits, cols):
    rng = np.random.default_rng(cols + bits)
    x = (0.01 * rng.random((11, cols))).astype(np.float32)
    x[1] += 0.2            # |min / s| 5e3 at 8 bits
    x[2] += 40.0           # 1e6: just below 2^20
    x[3] -= 42.0           # just above
    x[4] += 3000.0         # 8e7: the zero point is no longer exact to one
    ref = O.quantize_rtn(x, bits)
    q = {2: B.quantize_int2, 4: B.quantize_int4, 8: B.quantize_int8}[bits](f32_to_device(x))
    got = from_device_q(q)
    assert np.array_equal(got.scales, ref.scales) and np.array_equal(got.zeros, ref.zeros)
    assert np.array_equal(got.codes, ref.codes)
    assert np.array_equal(B.dequantize(q).cpu().numpy(), O.dequantize(ref))
    pad = q.codes[:, (cols * bits + 7) // 8:]             # what lies past the matrix holds code 0, as in an empty one
    assert torch.equal(pad, B.QTensor.empty(11, cols, bits).codes[:, (cols * bits + 7) // 8:])
