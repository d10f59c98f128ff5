"""K_b of kvq_drift_window at columns whose mean lies within 2^-48 of rho_K: the
column sums are fp64, so every such column falls on its side."""

import math

import numpy as np
import pytest
import torch

from paper_2607_16248_gb300 import kvq

pytestmark = pytest.mark.gpu


def columns(rows, k_max, rho, seed, margin):
    """Coverages in [0, 1] of very unequal size.  The mean of every column but
    the last is rho (1 - margin), of the last rho (1 + margin), exactly to a
    thousandth of the margin."""
    rng = np.random.default_rng(seed)
    c = (rng.random((rows, k_max)) ** 6).astype(np.float32)
    c *= np.float32(1.9 * rho) / c.mean(0)
    c = np.minimum(c, 1.0).astype(np.float32)
    for k in range(k_max):
        want = rows * rho * (1.0 + (margin if k == k_max - 1 else -margin))
        col = c[:, k]
        j = np.searchsorted(np.cumsum(col, dtype=np.float64), want - 3.0)
        col[j:] = 0.0  # the rest in up to eight single elements
        for i in range(rows - 8, rows):
            left = want - math.fsum(col.tolist())
            x = np.float32(min(left, 1.0))
            col[i] = x if float(x) <= left else np.nextafter(x, np.float32(0))
        assert j < rows - 8
        assert abs(math.fsum(col.tolist()) - want) < 1e-3 * want * margin
        rng.shuffle(col)
    return c


# fp64 sums of a thread's rows (at most 2048) round off by up to 2^-53 each, as
# a random walk of about 2^-51 of the sum; the margin is 2^-48
@pytest.mark.parametrize("rows,k_max", [(20480, 128), (65536, 256)])
def test_columns_next_to_rho(kvq_lib, rows, k_max):
    rho = float(np.float32(0.31))
    cov = columns(rows, k_max, rho, rows, 2.0 ** -48)
    kb, mean = kvq.drift_window(torch.from_numpy(cov).cuda(), rho)
    assert int(kb.item()) == k_max
    assert np.abs(mean.cpu().numpy() - np.float32(rho)).max() <= np.spacing(np.float32(rho))
