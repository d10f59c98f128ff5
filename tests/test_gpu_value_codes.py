"""Value codes in the MMA's operands (csrc/attn_core.cuh, Codes): with 1-bit keys
(exact operands) the error of fp32 attention results against 64 bits is what
the value accumulators lose.  Codes below the top of an fp16 number's low
eleven bits lose alignment bits there."""

import numpy as np
import pytest
import torch

import _util
from oracle import attention
from paper_2607_16248_gb300 import kvq, synth

pytestmark = pytest.mark.gpu


# The inputs are seeded and the results repeat.  With codes as fp16 integers
# (1024 + code, minus 1024), which lose nothing, the means are 1.17e-6 (groups
# of 4, 2 bits), 1.35e-6 (groups of 8, 2 bits) and 1.50e-6 (4 bits); codes one
# to six bits below the top give 1.61e-6, 1.66e-6 and 1.84e-6.
@pytest.mark.parametrize("bits,gq,bound", [(2, 4, 1.3e-6), (2, 8, 1.45e-6), (4, 8, 1.65e-6)])
def test_value_accumulators_keep_their_alignment(kvq_lib, bits, gq, bound):
    cfg = kvq.CacheConfig(batch=1, n_q_heads=8 * gq, n_kv_heads=8, bits_k=1, bits_v=bits,
                          max_len=2560)
    errs = []
    for seed in range(4):
        cache, kv = _util.make_cache(cfg, [2500], seed=seed)
        q = synth.queries(seed, 1, 8 * gq)
        out = kvq.kvq_decode_attn(cache, q.cuda(), out_dtype=torch.float32)
        out = out.cpu().double().numpy()[0]
        ref = attention.decode_attention(q[0].numpy(), _util.oracle_heads(cfg, *kv[0]))
        errs.append(np.linalg.norm(out - ref) / np.linalg.norm(ref))
    assert np.mean(errs) <= bound, errs
