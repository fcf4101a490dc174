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


@pytest.mark.parametrize("bits", [2, 4, 8])
def test_values_that_no_scale_brings_near_the_codes(bits):
    """A NaN takes the smallest code and no part in its group's extent; an infinity, or an extent past binary32's largest number,
    makes the group's scale its largest magnitude (1 if that is infinite), so that a scaled value can be anything."""
    rng = np.random.default_rng(bits)
    big = np.finfo(np.float32).max
    x = rng.standard_normal((8, 512)).astype(np.float32)
    x[0, ::7] = np.nan
    x[1, 200:] = np.nan                              # a group without a number, and part of the one before
    x[2, 3], x[2, 300] = np.inf, -np.inf
    x[3, 5], x[3, 6:60] = np.inf, -2.0e7             # scaled to below -1.5 * 2^23
    x[4, 5], x[4, 6:60] = -np.inf, 2.0e7
    x[5, :256] = np.linspace(-float(big), 1.1e31, 256)   # the extent overflows: scaled by the largest, to -3e7
    x[6, 17], x[6, 200] = np.nan, np.inf
    q = {2: B.quantize_int2, 4: B.quantize_int4, 8: B.quantize_int8}[bits](f32_to_device(x))
    got = from_device_q(q)
    lo, hi = np.float32(-(1 << (bits - 1))), np.float32((1 << (bits - 1)) - 1)
    with np.errstate(all="ignore"):
        for g in range(2):
            seg = x[:, 256 * g:256 * (g + 1)]
            ends = np.stack([np.fmin.reduce(seg, axis=1, initial=np.inf), np.fmax.reduce(seg, axis=1, initial=-np.inf)], axis=1)
            s, inv, z = O.group_params(ends.astype(np.float32), bits)
            assert np.array_equal(got.scales[:, g], s) and np.array_equal(got.zeros[:, g], z)
            code = np.fmin(np.fmax(np.rint(seg * inv[:, None]) + z[:, None], lo), hi)
            assert np.array_equal(got.codes[:, 256 * g:256 * (g + 1)], code.astype(np.int8))
