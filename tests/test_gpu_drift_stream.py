"""The drift metrics' streaming kernel at the edges of its rules: both block
sizes (launches of more and of fewer rows than SMs), rows at every 4-byte
alignment, logits its sample does not represent, candidate lists that
overflow, and rows it has to leave to the general kernel among others that it
settles.  Bounds are those of test_gpu_drift (float64 oracle)."""

import pytest
import torch

from paper_2607_16248_gb300 import kvq, synth
from test_gpu_drift import _compare

pytestmark = pytest.mark.gpu


def _kind(zf, zq, kind):
    """Rows of one kind: plain, one confident token far above the sample, the
    vocabulary in falling order, two levels, flat."""
    if kind == "peaky":
        zf[:, 1234 % zf.shape[1]] += 30.0
        zq[:, 1234 % zf.shape[1]] += 29.0
    elif kind == "sorted":
        zf, order = zf.sort(dim=-1, descending=True)
        zq = zq.gather(1, order)
    elif kind == "top_block":  # the best tokens side by side
        zf[:, 500:1500] += 6.0
        zq[:, 500:1500] += 6.0
    elif kind == "flat":
        zf, zq = zf * 1e-3, zq * 1e-3
    return zf.contiguous(), zq.contiguous()


@pytest.mark.parametrize("kind", ["plain", "peaky", "sorted", "top_block", "flat"])
@pytest.mark.parametrize("V,k_max", [(4099, 10), (8195, 16), (40001, 100), (131075, 256)])
def test_kinds(kvq_lib, kind, V, k_max):
    zf, zq = _kind(*synth.paired_logits(V + len(kind), 3, V, sigma=2.5, noise=0.4), kind)
    _compare(zf, zq, 0.9, 8, k_max, 0.02, 0.5, require=0.6)


@pytest.mark.parametrize("rows", [1, 152, 153, 700])
def test_row_counts(kvq_lib, rows):
    zf, zq = synth.paired_logits(rows, rows, 6001, sigma=2.0, noise=0.3)
    zf[::7] *= 1e-3  # rows for the general kernel in between
    zq[::7] *= 1e-3
    pick = sorted({0, 1, 6, 7, rows // 2, rows - 1} & set(range(rows)))
    _compare(zf, zq, 0.8, 4, 12, 0.02, 0.5, rows=pick, require=0.6)


@pytest.mark.parametrize("V", [40960, 40961, 131075, 163840])
def test_few_long_rows(kvq_lib, V):
    """Launches of few long rows go to the general kernel, longer ones (40
    rows: on either side of the rule for any SM count) to the streaming one:
    the same decisions and, the terms being the same integers, sums."""
    zf, zq = (z.cuda() for z in synth.paired_logits(V, 40, V, sigma=2.5, noise=0.4))
    whole = kvq.drift_metrics(zf, zq, 0.95, 8, 100, 0.02, 0.5)
    for lo, n in ((0, 1), (1, 16), (17, 17)):
        part = kvq.drift_metrics(zf[lo:lo + n], zq[lo:lo + n], 0.95, 8, 100, 0.02, 0.5)
        for k in ("m_t", "y_t", "c_t", "cov"):
            assert torch.equal(part[k], whole[k][lo:lo + n]), k
        # its sums of products run in another order: double-float rounding
        torch.testing.assert_close(part["d_loc"], whole["d_loc"][lo:lo + n], rtol=1e-6, atol=2e-7)
    _compare(zf[:2].cpu(), zq[:2].cpu(), 0.95, 8, 100, 0.02, 0.5, require=0.6)


@pytest.mark.parametrize("shift", [1, 2, 3])
def test_unaligned_rows(kvq_lib, shift):
    # each array's rows start at 4-byte alignments of their own
    zf, zq = synth.paired_logits(shift, 2, 9001)
    bufs = []
    for i, z in enumerate((zf, zq)):
        b = torch.empty(z.numel() + 8, device="cuda")
        v = b[shift + i:shift + i + z.numel()].view_as(z)
        v.copy_(z)
        bufs.append(v)
    a = kvq.drift_metrics(bufs[0], bufs[1], 0.9, 8, 20, 0.02, 0.5)
    b = kvq.drift_metrics(zf.cuda(), zq.cuda(), 0.9, 8, 20, 0.02, 0.5)
    assert torch.equal(a["m_t"], b["m_t"]) and torch.equal(a["y_t"], b["y_t"])
    # the sums run over the same terms in another order: 2^-40 and 2^-46 parts
    for k in ("c_t", "d_loc", "cov"):
        torch.testing.assert_close(a[k], b[k], rtol=0, atol=2e-6)


@pytest.mark.parametrize("rows,k_max", [(1, 1), (3, 256), (1025, 64), (70000, 7), (4097, 100)])
def test_window_means(kvq_lib, rows, k_max):
    g = synth.generator(rows)
    cov = torch.rand(rows, k_max, generator=g).cumsum(-1) / k_max
    kb, mean = kvq.drift_window(cov.cuda(), 0.31)
    want = cov.double().mean(0)
    # the fp32 rounding of the mean
    torch.testing.assert_close(mean.cpu().double(), want, rtol=1.2e-7, atol=0)
    hit = (want >= 0.3100000023841858).nonzero()
    assert int(kb.item()) == (int(hit[0]) + 1 if len(hit) else 0)
