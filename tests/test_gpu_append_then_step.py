"""A 32-token append that ends one token before a block boundary writes one page,
and the step behind it, which already plans while the append runs, pushes the
next block out of the window: the calls enqueued back to back leave the same
cache and results as with a wait after each."""

import pytest
import torch

from paper_2607_16248_gb300 import kvq, synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n_splits", [0, 1, 3])
@pytest.mark.parametrize("bits,paged", [(1, False), (2, True), (4, False), (8, True)])
def test_append_to_the_boundary_then_flush(kvq_lib, n_splits, bits, paged):
    cfg = kvq.CacheConfig(batch=2, n_q_heads=8, n_kv_heads=2, bits_k=bits, bits_v=bits,
                          max_len=1024)
    start, rounds = 223, 10  # 32 * 6 + 31
    n = start + 64 * rounds
    kv = [synth.kv_heads(80 + b, 2, n) for b in range(2)]
    k, v = (torch.stack([x[i] for x in kv]).cuda() for i in range(2))
    q = torch.stack([synth.queries(40 + i, 2, 8) for i in range(rounds)]).cuda()
    res = []
    for wait in (False, True):
        cache = kvq.QuantKVCache(cfg, n_pages=64 if paged else None)
        if paged:
            for b in range(2):
                cache.map_blocks(b, range(32), [(7 * (32 * b + j)) % 64 for j in range(32)])
        ws = kvq.attn_workspace(cfg, n_splits)
        parts, at = [], 0
        for c in [start] + [32, 1, 31] * rounds:
            parts.append([x[:, :, at:at + c].contiguous() for x in (k, v)])
            at += c
        outs = []
        torch.cuda.synchronize()
        for i, (a, b) in enumerate(parts):
            if a.shape[2] == 1:
                outs.append(kvq.kvq_decode_step(cache, a[:, :, 0].contiguous(),
                                                b[:, :, 0].contiguous(), q[i // 3],
                                                n_splits=n_splits, workspace=ws,
                                                out_dtype=torch.float32))
            else:
                kvq.kvq_pack(cache, a, b)
            if wait:
                torch.cuda.synchronize()
        torch.cuda.synchronize()
        assert cache.flags() == 0 and cache.seq_lens().tolist() == [n, n]
        nb = kvq.packed_len(n) // 32
        pages = torch.stack([cache.head_pages(b, h, nb) for b in range(2) for h in range(2)])
        res.append((torch.stack(outs), pages))
    (a, p), (b, r) = res
    assert torch.equal(p, r)
    rms = b.square().mean(-1, keepdim=True).sqrt()
    # the order of the fp32 sums is the plan's, made from the same lengths
    assert float(((a - b).abs() / rms).max()) <= 1e-5
