"""The flat plan behind a kernel that lets its dependents start early and only
then writes what a decode call reads: the block table, pages, the fp16 rings
(with a block that leaves the window in the call), lengths.  The results and
the cache are those of a call on the new contents, bit for bit."""

import ctypes
import subprocess

import pytest
import torch

from paper_2607_16248_gb300 import build, kvq, synth

pytestmark = pytest.mark.gpu

HELPER = r"""
#include <cstdint>
// Lets the next kernel of the stream start, waits about 60 us and copies n
// words.
__global__ void late_copy(uint32_t* dst, const uint32_t* src, long long n, long long cycles) {
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  const long long t0 = clock64();
  while (clock64() - t0 < cycles) {
  }
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n;
       i += (long long)gridDim.x * blockDim.x)
    dst[i] = src[i];
}
extern "C" int late_copy_on(void* dst, const void* src, long long words, void* stream) {
  late_copy<<<8, 256, 0, static_cast<cudaStream_t>(stream)>>>(
      static_cast<uint32_t*>(dst), static_cast<const uint32_t*>(src), words, 120000LL);
  return (int)cudaGetLastError();
}
"""


@pytest.fixture(scope="module")
def late_copy(tmp_path_factory, kvq_lib):
    d = tmp_path_factory.mktemp("late")
    src, so = d / "late.cu", d / "late.so"
    src.write_text(HELPER)
    subprocess.run([build._nvcc(), *build.ARCH, "-O2", "-shared", "-Xcompiler", "-fPIC", str(src),
                    "-o", str(so)], check=True, capture_output=True)
    fn = ctypes.CDLL(str(so)).late_copy_on
    fn.argtypes = [ctypes.c_void_p, ctypes.c_void_p, ctypes.c_longlong, ctypes.c_void_p]

    def run(dst, src):
        assert dst.is_contiguous() and src.is_contiguous()
        n = dst.numel() * dst.element_size()
        assert n == src.numel() * src.element_size() and n % 4 == 0
        assert fn(dst.data_ptr(), src.data_ptr(), n // 4,
                  torch.cuda.current_stream().cuda_stream) == 0
    return run


HKV, HQ = 2, 8


def _cfg(bits, batch):
    return kvq.CacheConfig(batch=batch, n_q_heads=HQ, n_kv_heads=HKV, bits_k=bits, bits_v=bits,
                           max_len=1024)


def _fill(cfg, L, seed):
    cache = kvq.QuantKVCache(cfg)
    for ring in cache.resid():
        ring.zero_()
    cache.pages().zero_()
    for b in range(cfg.batch):
        k, v = synth.kv_heads(seed + b, HKV, L)
        kvq.kvq_pack(cache, k[None].cuda(), v[None].cuda(), batch_begin=b)
    return cache


def _call(cache, step, seed):
    cfg = cache.cfg
    q = synth.queries(seed, cfg.batch, HQ).cuda()
    ws = kvq.attn_workspace(cfg, 0)
    g = synth.generator(seed + 1)
    kn, vn = (torch.randn(cfg.batch, HKV, 128, generator=g).half().cuda() for _ in range(2))
    out = torch.empty(q.shape, dtype=torch.float32, device="cuda")
    torch.cuda.synchronize()

    def go():
        if step:
            kvq.kvq_decode_step(cache, kn, vn, q, out=out, n_splits=0, workspace=ws)
        else:
            kvq.kvq_decode_attn(cache, q, out=out, n_splits=0, workspace=ws)
        return out
    return go


# 703 and 671 tokens: a step pushes a block out of the window (32 k + 128 - 1)
# (703 = 32 * 18 + 127, 671 = 32 * 17 + 127)
@pytest.mark.parametrize("what", ["pages", "rings", "both"])
@pytest.mark.parametrize("bits,L,step", [(2, 703, False), (2, 703, True), (1, 703, True),
                                         (4, 671, True), (8, 700, True)])
def test_contents_written_late(kvq_lib, late_copy, what, bits, L, step):
    cfg = _cfg(bits, 3)
    old, new, ref = (_fill(cfg, L, s) for s in (10, 50, 50))
    lo, hi = {"pages": (0, 1), "rings": (1, 3), "both": (0, 3)}[what]
    a, b = cfg.layout()[1][lo], cfg.layout()[1][hi]
    # the reference: what the caller means the cache to be
    ref.buffer.copy_(old.buffer)
    ref.buffer[a:b].copy_(new.buffer[a:b])
    want = _call(ref, step, 5)().clone()
    go = _call(old, step, 5)
    late_copy(old.buffer[a:b], new.buffer[a:b])
    got = go()
    torch.cuda.synchronize()
    assert old.flags() == 0 and torch.equal(got, want)
    assert torch.equal(old.buffer, ref.buffer)


@pytest.mark.parametrize("step", [False, True])
def test_table_written_late(kvq_lib, late_copy, step):
    """The table moves to other page sets; before, it maps to none in part."""
    cfg, L, n = _cfg(2, 1), 703, 24
    cache = kvq.QuantKVCache(cfg, n_pages=2 * n)
    tables = []
    for first in (0, n):  # the same window, other blocks
        k, v = synth.kv_heads(first + 3, HKV, L)
        kw, vw = synth.kv_heads(99, HKV, L)
        k[:, L - 200:], v[:, L - 200:] = kw[:, L - 200:], vw[:, L - 200:]
        cache.reset()
        cache.map_blocks(0, range(n), [first + (5 * j) % n for j in range(n)])
        kvq.kvq_pack(cache, k[None].cuda(), v[None].cuda())
        tables.append(cache.block_table.clone())
    lens = cache.seq_lens().clone()
    go = _call(cache, step, 6)
    want = go().clone()  # tables[1]
    cache.seq_lens().copy_(lens)
    for before in (tables[0], torch.full_like(tables[0], -1)):
        cache.block_table.copy_(before)
        torch.cuda.synchronize()
        late_copy(cache.block_table, tables[1])
        got = go()
        torch.cuda.synchronize()
        assert cache.flags() == 0 and torch.equal(got, want)
        cache.seq_lens().copy_(lens)


@pytest.mark.parametrize("lens", [[703, 0, 130], [671, 699, 20], [0, 0, 0]])
def test_lengths_written_late(kvq_lib, late_copy, lens):
    cfg = _cfg(2, 3)
    cache = _fill(cfg, 703, 30)
    live = cache.seq_lens()
    new = torch.tensor(lens, dtype=torch.int32, device="cuda")
    start = live.clone()
    go = _call(cache, False, 7)
    live.copy_(new)
    want = go().clone()
    live.copy_(start)
    torch.cuda.synchronize()
    late_copy(live, new)
    got = go()
    torch.cuda.synchronize()
    assert cache.flags() == 0 and torch.equal(got, want)
