"""Rows that the streaming kernel leaves to the general one, or that go to it
alone: alpha = 1 at narrow and wide logits (the boundary inside and below the
histogram), logits closer together than its lists hold, in launches of fewer
and of more rows than the GPU runs clusters at once."""

import pytest
import torch

from paper_2607_16248_gb300 import kvq, synth
from test_gpu_drift import _compare

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("rows", [3, 47, 170])
@pytest.mark.parametrize("sigma,alpha", [(0.002, 0.9), (0.02, 0.5), (1.0, 1.0), (3.0, 1.0)])
@pytest.mark.parametrize("V", [3001, 30000])
def test_left_rows(kvq_lib, rows, sigma, alpha, V):
    zf, zq = synth.paired_logits(rows + V, rows, V, sigma=sigma, noise=0.1 * sigma)
    if rows == 170:
        zf[:, 5::11] = float("-inf")  # masked tokens
        zq[:, 5::11] = float("-inf")
    pick = sorted({0, rows // 2, rows - 1})
    # alpha = 1 asks for the last token whose mass is not nothing in fp32,
    # which float64 has another of: only the shares are compared there
    if alpha < 1.0:
        _compare(zf, zq, alpha, 8, 32, 0.02, 0.5, rows=pick, require=0.3)
    a = kvq.drift_metrics(zf.cuda(), zq.cuda(), alpha, 8, 32, 0.02, 0.5)
    for r in pick:  # alone: the same bits
        b = kvq.drift_metrics(zf[r:r + 1].cuda(), zq[r:r + 1].cuda(), alpha, 8, 32, 0.02, 0.5)
        for k in a:
            assert torch.equal(a[k][r:r + 1], b[k]), (k, r)
    if alpha == 1.0:
        top = zq.topk(32, dim=-1).indices
        cov = torch.softmax(zf.double(), -1).gather(1, top).cumsum(-1)
        assert float((a["cov"].cpu().double() - cov).abs().max()) <= 2e-6
