"""Decode attention at the edges of its window units (16 tokens staged at once,
or 32-token chunks on long ranges of the split plan), of its code operands
(2- and 4-bit codes in subnormal fp16 numbers) and of the plan that is made
before the dependency wait.  Bounds: 2e-3 of the per-head rms against the
float64 oracle (test_gpu_attn); tighter ones are derived where they stand."""

import numpy as np
import pytest
import torch

import _util
from oracle import attention
from paper_2607_16248_gb300 import kvq, synth
from test_gpu_attn import _run

pytestmark = pytest.mark.gpu

EDGES = [1, 15, 16, 17, 31, 33, 48, 127, 129, 143, 144, 145, 159, 160, 161, 176, 193]


@pytest.mark.parametrize("bk,bv,gq", [(2, 2, 4), (4, 4, 5), (1, 1, 3), (8, 2, 8)])
@pytest.mark.parametrize("n_splits", [0, 1, 3])
def test_window_lengths_around_units(kvq_lib, bk, bv, gq, n_splits):
    cfg = kvq.CacheConfig(batch=len(EDGES), n_q_heads=gq, n_kv_heads=1, bits_k=bk, bits_v=bv,
                          max_len=224)
    errs, _ = _run(cfg, EDGES, seed=11 * bk + bv, n_splits=n_splits)
    assert errs.max() <= _util.ATTN_TOL, errs.max(axis=1)


@pytest.mark.parametrize("n_splits,L", [(1, 1151), (1, 1152), (1, 1153), (1, 1185), (2, 2177)])
def test_ranges_at_the_chunk_rule(kvq_lib, n_splits, L):
    # 16 n_splits warps: two blocks per warp is the last range with 16-token
    # units (nb = 32 n_splits), one block more the first with 32-token chunks
    cfg = kvq.CacheConfig(batch=1, n_q_heads=5, n_kv_heads=1, bits_k=2, bits_v=4, max_len=2304)
    errs, _ = _run(cfg, [L], seed=L, n_splits=n_splits)
    assert errs.max() <= _util.ATTN_TOL


@pytest.mark.parametrize("residual", [32, 288])
@pytest.mark.parametrize("n_splits", [0, 1])
def test_other_window_sizes(kvq_lib, residual, n_splits):
    cfg = kvq.CacheConfig(batch=2, n_q_heads=4, n_kv_heads=1, bits_k=2, bits_v=2, max_len=1024,
                          residual=residual)
    errs, _ = _run(cfg, [1000, residual + 17], seed=residual, n_splits=n_splits)
    assert errs.max() <= _util.ATTN_TOL


@pytest.mark.parametrize("bits", [2, 4])
@pytest.mark.parametrize("gq", [1, 4, 5, 8])
def test_subnormal_code_operands_lose_nothing(kvq_lib, bits, gq):
    # fp32 results: a score's partial sums (up to ~64 in the log2 domain) are
    # kept to 2^-24 over 8 accumulations, 3e-5 at worst per score and an
    # order less in the sums over tokens; codes left at the bottom of a
    # subnormal number's mantissa give 2e-4
    cfg = kvq.CacheConfig(batch=1, n_q_heads=gq, n_kv_heads=1, bits_k=bits, bits_v=bits,
                          max_len=3072)
    cache, kv = _util.make_cache(cfg, [3000], seed=gq)
    q = synth.queries(gq, 1, gq)
    out = kvq.kvq_decode_attn(cache, q.cuda(), out_dtype=torch.float32).cpu().double().numpy()[0]
    ref = attention.decode_attention(q[0].numpy(), _util.oracle_heads(cfg, *kv[0]))
    assert np.linalg.norm(out - ref) <= 1e-5 * np.linalg.norm(ref)


@pytest.mark.parametrize("n_splits", [0, 2])
@pytest.mark.parametrize("paged", [False, True])
def test_steps_enqueued_back_to_back(kvq_lib, n_splits, paged):
    """Every step's lengths change while the next launch is already planning:
    70 steps of one cache in a row, two of its sequences flushing on the way,
    against kvq_pack and kvq_decode_attn with a wait between."""
    cfg = kvq.CacheConfig(batch=3, n_q_heads=8, n_kv_heads=2, bits_k=2, bits_v=2, max_len=512)
    start, steps = [300, 1, 130], 70
    kv = [synth.kv_heads(5 + b, 2, start[b] + steps) for b in range(3)]
    q = torch.stack([synth.queries(90 + i, 3, 8) for i in range(steps)]).cuda()
    outs = []
    for fused in (True, False):
        cache = kvq.QuantKVCache(cfg, n_pages=48 if paged else None)
        if paged:
            for b in range(3):
                cache.map_blocks(b, range(16), [(5 * (16 * b + j)) % 48 for j in range(16)])
        for b, (k, v) in enumerate(kv):
            kvq.kvq_pack(cache, k[:, :start[b]][None].contiguous().cuda(),
                         v[:, :start[b]][None].contiguous().cuda(), batch_begin=b)
        ws = kvq.attn_workspace(cfg, n_splits)
        new = [[torch.stack([kv[b][j][:, start[b] + i] for b in range(3)]).contiguous().cuda()
                for j in range(2)] for i in range(steps)]
        torch.cuda.synchronize()
        got = []
        for i in range(steps):
            if fused:
                got.append(kvq.kvq_decode_step(cache, *new[i], q[i], n_splits=n_splits, workspace=ws,
                                               out_dtype=torch.float32))
            else:
                kvq.kvq_pack(cache, new[i][0][:, :, None].contiguous(),
                             new[i][1][:, :, None].contiguous())
                torch.cuda.synchronize()
                got.append(kvq.kvq_decode_attn(cache, q[i], n_splits=n_splits, workspace=ws,
                                               out_dtype=torch.float32))
                torch.cuda.synchronize()
        torch.cuda.synchronize()
        assert cache.flags() == 0 and cache.seq_lens().tolist() == [s + steps for s in start]
        outs.append(torch.stack(got))
    a, b = outs
    rms = b.square().mean(-1, keepdim=True).sqrt()
    # the two paths differ by fp32 summation order
    assert float(((a - b).abs() / rms).max()) <= 1e-4


@pytest.mark.parametrize("bits", [1, 4])
def test_flushing_step_behind_a_long_append(kvq_lib, bits):
    """Every step flushes a block whose ring rows the append just before it
    wrote (95 tokens, then one step, five times): the same lengths and
    results with the calls enqueued back to back as with a wait after each."""
    cfg = kvq.CacheConfig(batch=2, n_q_heads=8, n_kv_heads=2, bits_k=bits, bits_v=bits,
                          max_len=512, residual=32)
    kv = [synth.kv_heads(60 + b, 2, 480) for b in range(2)]
    k, v = (torch.stack([kv[b][j] for b in range(2)]).cuda() for j in range(2))
    q = torch.stack([synth.queries(70 + i, 2, 8) for i in range(5)]).cuda()
    packs = [[x[:, :, 96 * i:96 * i + 95].contiguous() for x in (k, v)] for i in range(5)]
    news = [[x[:, :, 96 * i + 95].contiguous() for x in (k, v)] for i in range(5)]
    res = []
    for wait in (False, True):
        cache = kvq.QuantKVCache(cfg)
        ws = kvq.attn_workspace(cfg, 0)
        torch.cuda.synchronize()
        outs = []
        for i in range(5):
            kvq.kvq_pack(cache, *packs[i])
            if wait:
                torch.cuda.synchronize()
            outs.append(kvq.kvq_decode_step(cache, *news[i], q[i], n_splits=0, workspace=ws,
                                            out_dtype=torch.float32))
            if wait:
                torch.cuda.synchronize()
        torch.cuda.synchronize()
        assert cache.flags() == 0 and cache.seq_lens().tolist() == [480, 480]
        # once more over all the blocks
        outs.append(kvq.kvq_decode_attn(cache, q[0], n_splits=1, workspace=kvq.attn_workspace(cfg, 1),
                                        out_dtype=torch.float32))
        res.append(torch.stack(outs))
    # partials merge in an order that may differ between runs: fp32 rounding
    a, b = res
    rms = b.square().mean(-1, keepdim=True).sqrt()
    assert float(((a - b).abs() / rms).max()) <= 1e-5
