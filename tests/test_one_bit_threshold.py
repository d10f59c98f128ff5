"""The 1-bit quantizer's fp16 threshold (csrc/common.cuh, threshold_codes)
against the oracle's definition (oracle/quant.py): code = x > t, t found from
RN16(RN32(zero + scale / 2)) and one neighbour.  Groups where that pair of
tests does not settle t go to the general steps; on all others every code
must agree."""

import numpy as np
import pytest

from oracle import quant
from test_quant_shortcuts import _groups

F32 = np.float32


def _order(h):
    b = h.view(np.int16).astype(np.int32)
    return np.where(b < 0, -(b & 0x7FFF), b)


def _half(k):
    return np.where(k < 0, (-k) | 0x8000, k).astype(np.uint16).view(np.float16)


def _threshold_codes(x):
    _, scale, zero = quant.quantize_groups(x, 1)
    lo = zero.astype(F32)
    b = scale.astype(F32) * F32(0.5)

    def below(k):
        return (_half(k).astype(F32) - lo).astype(F32) <= b

    k = _order((lo + b).astype(F32).astype(np.float16))
    at = below(k)
    k = np.where(at, k, k - 1)
    settled = np.where(at, ~below(k + 1), below(k))
    return (x > _half(k)[..., None]).astype(np.uint8), settled


@pytest.mark.parametrize("seed", [1, 2])
def test_settled_groups_match_the_definition(seed):
    x = _groups(np.random.default_rng(seed), 1, 50000)
    want, _, _ = quant.quantize_groups(x, 1)
    got, settled = _threshold_codes(x)
    assert np.array_equal(got[settled], want[settled])
    assert 0.99 < settled.mean() < 1.0  # some are left, and they are rare


def test_few_values_two_levels_and_constants():
    rng = np.random.default_rng(3)
    base = rng.standard_normal((20000, 1))
    step = 2.0 ** rng.integers(-14, 3, (20000, 1))
    x = np.clip(base + step * rng.integers(0, 3, (20000, 32)), -6e4, 6e4).astype(np.float16)
    x[::5] = x[::5, :1]  # constant groups: scale 0, code 0
    want, _, _ = quant.quantize_groups(x, 1)
    got, settled = _threshold_codes(x)
    assert np.array_equal(got[settled], want[settled]) and settled.mean() > 0.99
