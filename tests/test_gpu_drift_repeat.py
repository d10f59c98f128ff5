"""A row's drift metrics depend on nothing but the row: the same bits in every
run, in launches of any number of rows (which take different kernels and block
sizes) and at any place among them."""

import pytest
import torch

from paper_2607_16248_gb300 import kvq, synth

pytestmark = pytest.mark.gpu
KEYS = ("m_t", "c_t", "d_loc", "y_t", "cov")


def _run(zf, zq, alpha, k_max):
    o = kvq.drift_metrics(zf, zq, alpha, 8, k_max, 0.02, 0.5)
    torch.cuda.synchronize()
    return o


@pytest.mark.parametrize("V,alpha,k_max", [(3001, 0.9, 16), (9004, 0.99, 64), (50001, 0.9, 100),
                                           (50001, 0.99, 256)])
def test_any_launch_gives_the_same_bits(kvq_lib, V, alpha, k_max):
    rows = 200
    # close pairs: d_loc is what is left of sums near 1, so that a change in
    # their last bits shows
    zf, zq = (z.cuda() for z in synth.paired_logits(V, rows, V, sigma=2.5, noise=2e-5))
    zf[5] *= 1e-3  # a row for the general kernel among the others
    zq[5] *= 1e-3
    whole = _run(zf, zq, alpha, k_max)
    for _ in range(3):
        again = _run(zf, zq, alpha, k_max)
        for k in KEYS:
            assert torch.equal(whole[k], again[k]), k
    for lo, n in ((0, 1), (3, 7), (10, 15), (20, 16), (30, 152)):
        part = _run(zf[lo:lo + n], zq[lo:lo + n], alpha, k_max)
        for k in KEYS:
            assert torch.equal(part[k], whole[k][lo:lo + n]), (k, lo, n)


def test_close_rows_keep_their_difference(kvq_lib):
    """z_q next to z_fp: d_loc is what is left of sums near 1 that cancel.  The
    product sums are good to 2^-50 of them and the masses to 2^-40 a term, so
    a distance of 1e-5 has an error well below 1e-3 of it; the terms' own fp32
    rounding (2^-23) is the rest."""
    V = 9001
    zf = synth.paired_logits(1, 4, V, sigma=2.5)[0].double()
    zq = (zf + 1e-4 * torch.randn(4, V, generator=synth.generator(9), dtype=torch.float64)).float()
    zf = zf.float()
    o = _run(zf.cuda(), zq.cuda(), 0.9, 16)
    a, b = zf.double(), zq.double()
    for r in range(4):
        order = a[r].argsort(descending=True, stable=True)[:int(o["m_t"][r])]
        top = b[r].argsort(descending=True, stable=True)[:8]
        u = torch.unique(torch.cat([order, top]))
        x, y = torch.softmax(a[r][u], 0), torch.softmax(b[r][u], 0)
        d = float((x - y).norm())
        assert 1e-7 < d < 1e-4
        assert abs(float(o["d_loc"][r]) - d) <= 2e-2 * d + 2e-7
