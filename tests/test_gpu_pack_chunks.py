"""Chunked prefill (Sec. 3.1): blocks that begin in the fp16 window and end in
the new tokens are quantized beside the others.  The cache after any chunking
equals the cache after one call, byte for byte, for chunk lengths around the
block and window sizes, every code width and windows of other lengths."""

import pytest
import torch

from paper_2607_16248_gb300 import kvq, synth

pytestmark = pytest.mark.gpu


def _filled(cfg, k, v, chunks, paged):
    cache = kvq.QuantKVCache(cfg, n_pages=cfg.batch * cfg.max_blocks if paged else None)
    if paged:
        n = cfg.max_blocks
        for b in range(cfg.batch):
            cache.map_blocks(b, range(n), [(b * n + 7 * j) % (cfg.batch * n) for j in range(n)]
                             if cfg.batch == 1 else [b * n + j for j in range(n)])
    for ring in cache.resid():
        ring.zero_()
    at = 0
    for c in chunks:
        kvq.kvq_pack(cache, k[:, :, at:at + c].contiguous(), v[:, :, at:at + c].contiguous())
        at += c
    torch.cuda.synchronize()
    assert cache.flags() == 0 and cache.seq_lens().tolist() == [at] * cfg.batch
    return cache


def _window(cache, L):
    cfg = cache.cfg
    slots = torch.arange(kvq.packed_len(L, cfg.residual), L, device="cuda") % cfg.ring
    return [r[:, :, slots] for r in cache.resid()]


@pytest.mark.parametrize("bits", [(1, 1), (2, 2), (4, 4), (8, 8), (2, 1), (1, 8)])
@pytest.mark.parametrize("chunk", [33, 63, 64, 95, 127, 160, 161, 300])
@pytest.mark.parametrize("residual,paged", [(128, False), (32, False), (64, True)])
def test_any_chunking_gives_the_same_cache(kvq_lib, bits, chunk, residual, paged):
    batch, hkv, L = 2, 2, 700
    cfg = kvq.CacheConfig(batch=batch, n_q_heads=hkv, n_kv_heads=hkv, bits_k=bits[0],
                          bits_v=bits[1], max_len=736, residual=residual)
    kv = [synth.kv_heads(7 * chunk + b, hkv, L) for b in range(batch)]
    k, v = (torch.stack([x[i] for x in kv]).cuda() for i in range(2))
    one = _filled(cfg, k, v, [L], paged)
    many = _filled(cfg, k, v, [min(chunk, L - a) for a in range(0, L, chunk)], paged)
    nb = kvq.packed_len(L, residual) // 32
    for b in range(batch):
        for h in range(hkv):
            assert torch.equal(one.head_pages(b, h, nb), many.head_pages(b, h, nb))
    for x, y in zip(_window(one, L), _window(many, L)):
        assert torch.equal(x, y)


def test_one_bit_codes_of_nan(kvq_lib):
    """A NaN among finite numbers gets the same 1-bit code in a long call (the
    threshold) as in short ones (the definition's arithmetic): equal bytes."""
    cfg = kvq.CacheConfig(batch=1, n_q_heads=2, n_kv_heads=2, bits_k=1, bits_v=1, max_len=256,
                          residual=32)
    g = torch.Generator().manual_seed(8)
    k, v = (torch.randn(1, 2, 224, 128, generator=g).half() for _ in range(2))
    for x in (k, v):
        x[torch.rand(x.shape, generator=g) < 0.02] = float("nan")
    pages = []
    for step in (224, 7):
        cache = kvq.QuantKVCache(cfg)
        for i in range(0, 224, step):
            kvq.kvq_pack(cache, k[:, :, i:i + step].contiguous().cuda(),
                         v[:, :, i:i + step].contiguous().cuda())
        torch.cuda.synchronize()
        pages.append(cache.pages()[:, :, :6].cpu())
    assert torch.equal(*pages)
