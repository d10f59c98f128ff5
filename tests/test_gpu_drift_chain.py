"""kvq_drift_window behind kvq_drift_metrics on one stream: the window kernel
starts before the metrics are written and reads them after its dependency
wait.  Every call of a chain on one set of outputs sees that step's coverage
and not the one before it."""

import pytest
import torch

from paper_2607_16248_gb300 import kvq, synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("rows,V,k_max", [(4, 3001, 16), (40, 9001, 256), (300, 4099, 256)])
def test_window_sees_this_steps_coverage(kvq_lib, rows, V, k_max):
    steps = 12
    z = []
    for i in range(steps):
        zf, zq = synth.paired_logits(i, rows, V, sigma=1.5 + 0.2 * i, noise=0.4)
        z.append((zf.cuda(), zq.cuda()))
    o = kvq.drift_metrics(*z[0], 0.9, 8, k_max, 0.02, 0.5)
    for i in range(steps):  # warm: lines of the old coverage in every cache
        kvq.drift_window(o["cov"], 0.5)
    torch.cuda.synchronize()
    chain = []
    for a, b in z:
        kvq.drift_metrics(a, b, 0.9, 8, k_max, 0.02, 0.5, outputs=o)
        chain.append(kvq.drift_window(o["cov"], 0.5))
    torch.cuda.synchronize()
    for (a, b), (kb, mean) in zip(z, chain):
        cov = kvq.drift_metrics(a, b, 0.9, 8, k_max, 0.02, 0.5)["cov"]
        torch.cuda.synchronize()
        kb2, mean2 = kvq.drift_window(cov, 0.5)
        assert torch.equal(mean, mean2) and torch.equal(kb, kb2)
