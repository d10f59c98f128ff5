"""The workloads whose speed is tracked: what each one stands for, its inputs,
one pass through the public entry points, the work it cannot do without and
the tolerance of its results.

Five kinds of case:

* ``step``     one decode step of a stack of attention layers: per layer one
               ``kvq_decode_step`` (append the token, quantize what leaves the
               window, attend), captured once in a CUDA graph and replayed, as
               a serving loop does.  Every pass decodes the same position: the
               lengths are set back inside the graph.
* ``attn``     the same stack through ``kvq_decode_attn`` (no append), for
               several queries over one prefix.
* ``prefill``  a slot is reset and a context packed into it by ``kvq_pack``,
               in one call or in chunks.
* ``dgap``     the epilogue of a decode step: the logits arrive (a copy stands
               for the LM head) and ``dgap_restore`` corrects them, as a graph.
* ``drift``    offline calibration on paired logits: ``kvq_drift_metrics`` and
               the window rule ``kvq_drift_window``.
"""

import random

import torch

from paper_2607_16248_gb300 import kvq

D = 128        # head size
G = 32         # tokens (keys) or channels (values) of a quantization group
DEV = "cuda"


def listed():
    return [
        # one user, short context, two-bit cache: launch and merge latency
        dict(name="step_b1_4k_k2v2", kind="step", batch=1, hq=32, hkv=8, bk=2, bv=2, ctx=4099,
             lo=4099, lens=0, layers=8, paged=False, f32=False),
        # one user, long chat, one-bit cache
        dict(name="step_b1_32k_k1v1", kind="step", batch=1, hq=32, hkv=8, bk=1, bv=1, ctx=32767,
             lo=32767, lens=0, layers=8, paged=False, f32=False),
        # one user, a whole-document context, four-bit cache
        dict(name="step_b1_128k_k4v4", kind="step", batch=1, hq=32, hkv=8, bk=4, bv=4, ctx=131010,
             lo=131010, lens=0, layers=4, paged=False, f32=False),
        # a serving batch with contexts of its own each, on paged blocks
        dict(name="step_b16_ragged_k2v2_paged", kind="step", batch=16, hq=32, hkv=8, bk=2, bv=2,
             ctx=32768, lo=8192, lens=4, layers=4, paged=True, f32=False),
        # a batch of long contexts, query groups of five: the benchmark's layer
        dict(name="step_b8_64k_k1v1_g5", kind="step", batch=8, hq=40, hkv=8, bk=1, bv=1,
             ctx=65536, lo=65536, lens=0, layers=4, paged=False, f32=False),
        # a small batch over a mid-sized prefix, eight-bit cache, query groups
        # of eight, fp32 results
        dict(name="attn_b4_16k_k8v8_g8_f32", kind="attn", batch=4, hq=64, hkv=8, bk=8, bv=8,
             ctx=16389, lo=16389, lens=0, layers=4, paged=False, f32=True),
        # prompts packed at once, a batch of long ones: the largest case
        dict(name="prefill_b8_64k_k1v1", kind="prefill", batch=8, hkv=8, bk=1, bv=1, ctx=65536,
             chunk=65536),
        # prompts that arrive in odd chunks, four-bit cache
        dict(name="prefill_b4_30k_chunked_k4v4", kind="prefill", batch=4, hkv=8, bk=4, bv=4,
             ctx=30011, chunk=4099),
        # one row of a 128k vocabulary, corrector always on: the latency of a
        # step's tail
        dict(name="dgap_b1_v128256", kind="dgap", batch=1, vocab=128256, k=32, hidden=256,
             tau=0.0),
        # a batch of rows of the largest vocabulary
        dict(name="dgap_b8_v152064", kind="dgap", batch=8, vocab=152064, k=32, hidden=256,
             tau=0.5),
        # a calibration trace: 256 steps of a 128k vocabulary
        dict(name="drift_256x128256", kind="drift", rows=256, vocab=128256, alpha=0.9, window=32,
             kmax=256, sigma=3.0, noise=0.4),
        # a short trace of a 32k vocabulary
        dict(name="drift_24x32003", kind="drift", rows=24, vocab=32003, alpha=0.95, window=16,
             kmax=64, sigma=2.5, noise=0.4),
    ]


def _log(rng, lo, hi):
    """A whole number spread over [lo, hi] by its logarithm."""
    return max(lo, min(hi, int(round(lo * (hi / lo) ** rng.random()))))


def draw(rng):
    kind = rng.choice(["step", "step", "step", "attn", "prefill", "dgap", "drift"])
    if kind in ("step", "attn"):
        layers = 4
        hkv = rng.choice([2, 4, 8, 8])
        bk = rng.choice([1, 2, 4, 8])
        bv = bk if rng.random() < 0.7 else rng.choice([1, 2, 4, 8])
        batch = _log(rng, 1, 24)
        # at most about the bytes of the largest listed cache
        cap = 1.0e9 / (layers * batch * hkv * (16 * (bk + bv) + 32))
        ctx = _log(rng, 300, int(max(600, min(131072, cap))))
        lo = ctx if batch == 1 or rng.random() < 0.5 else max(1, ctx // 4)
        return dict(kind=kind, batch=batch, hq=hkv * rng.choice([1, 2, 4, 5, 7, 8]), hkv=hkv,
                    bk=bk, bv=bv, ctx=ctx, lo=lo, lens=rng.randrange(1000), layers=layers,
                    paged=rng.random() < 0.3, f32=rng.random() < 0.3)
    if kind == "prefill":
        bits = rng.choice([1, 2, 4, 8])
        hkv = rng.choice([2, 4, 8])
        batch = _log(rng, 1, 8)
        ctx = _log(rng, 1000, 131072 if batch * hkv <= 32 else 65536)
        chunk = ctx if rng.random() < 0.5 else max(500, ctx // rng.randint(2, 6))
        return dict(kind=kind, batch=batch, hkv=hkv, bk=bits,
                    bv=bits if rng.random() < 0.7 else rng.choice([1, 2, 4, 8]), ctx=ctx,
                    chunk=chunk)
    if kind == "dgap":
        return dict(kind=kind, batch=_log(rng, 1, 32), vocab=_log(rng, 2000, 160000),
                    k=rng.choice([8, 16, 32, 32, 64]), hidden=rng.choice([64, 256, 256, 512]),
                    tau=rng.choice([0.0, 0.5, 0.6]))
    kmax = rng.choice([16, 64, 100, 256])
    return dict(kind=kind, rows=_log(rng, 4, 256), vocab=_log(rng, 2000, 160000),
                alpha=rng.choice([0.8, 0.9, 0.95, 0.99]), window=rng.choice([8, 16]), kmax=kmax,
                sigma=rng.uniform(2.0, 4.0), noise=rng.uniform(0.2, 0.6))


# ---------------------------------------------------------------------------
# Inputs
# ---------------------------------------------------------------------------


def _gen(*parts):
    s = 0
    for p in parts:
        s = (s * 1000003 + int(p) + 17) % (1 << 62)
    g = torch.Generator(device=DEV)
    g.manual_seed(s)
    return g


def _lengths(c):
    if c["lo"] >= c["ctx"]:
        return [c["ctx"]] * c["batch"]
    r = random.Random(c["lens"])
    return [r.randint(c["lo"], c["ctx"]) for _ in range(c["batch"])]


def _kv(g, lead, n):
    """Keys and values [*lead, n, 128]: normal, with four channels of every
    key head ten times as large (what makes low-bit keys hard)."""
    k = torch.randn(*lead, n, D, generator=g, device=DEV).half()
    v = torch.randn(*lead, n, D, generator=g, device=DEV).half()
    outlier = torch.rand(*lead, D, generator=g, device=DEV).argsort(-1) < 4
    return torch.where(outlier.unsqueeze(-2), k * 10, k), v


def _layer_kv(c, seed, layer, b, n):
    return _kv(_gen(seed, 1, layer, b), (c["hkv"],), n)


def _token(c, seed):
    g = _gen(seed, 2)
    q = torch.randn(c["layers"], c["batch"], c["hq"], D, generator=g, device=DEV).half()
    kn = torch.randn(c["layers"], c["batch"], c["hkv"], D, generator=g, device=DEV).half()
    vn = torch.randn(c["layers"], c["batch"], c["hkv"], D, generator=g, device=DEV).half()
    return q, kn, vn


def _dgap_weights(c, seed):
    g = _gen(seed, 3)
    k, h = c["k"], c["hidden"]
    nin = 5 * k + 8

    def u(shape, fan):
        return (torch.rand(*shape, generator=g, device=DEV) * 2 - 1) / fan ** 0.5

    return dict(det_w1=u((h, 8), 8), det_b1=u((h,), 8), det_w2=u((h,), h), det_b2=u((1,), h),
                cor_w1=u((h, nin), nin), cor_b1=u((h,), nin), cor_w2=u((k, h), h),
                cor_b2=u((k,), h))


def _logits(c, seed):
    return torch.randn(c["batch"], c["vocab"], generator=_gen(seed, 4), device=DEV) * 3


def _paired(c, seed):
    g = _gen(seed, 5)
    zf = torch.randn(c["rows"], c["vocab"], generator=g, device=DEV) * c["sigma"]
    return zf, zf + torch.randn(c["rows"], c["vocab"], generator=g, device=DEV) * c["noise"]


# ---------------------------------------------------------------------------
# States
# ---------------------------------------------------------------------------


def _capture(work):
    side = torch.cuda.Stream()
    side.wait_stream(torch.cuda.current_stream())
    with torch.cuda.stream(side):
        work()
    torch.cuda.current_stream().wait_stream(side)
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        work()
    return graph


def _prepare_decode(c, seed):
    lens = _lengths(c)
    step = c["kind"] == "step"
    # room to grow, as a server reserves
    cfg = kvq.CacheConfig(batch=c["batch"], n_q_heads=c["hq"], n_kv_heads=c["hkv"],
                          bits_k=c["bk"], bits_v=c["bv"], max_len=32 * (max(lens) // 32 + 16))
    nbs = [kvq.packed_len(n + step) // G for n in lens]
    caches = []
    for layer in range(c["layers"]):
        if c["paged"]:
            cache = kvq.QuantKVCache(cfg, DEV, n_pages=max(1, sum(nbs)))
            order = torch.randperm(max(1, sum(nbs)), generator=torch.Generator().manual_seed(
                seed * 64 + layer)).tolist()
            at = 0
            for b, nb in enumerate(nbs):
                if nb:
                    cache.map_blocks(b, range(nb), order[at:at + nb])
                at += nb
        else:
            cache = kvq.QuantKVCache(cfg, DEV)
        for ring in cache.resid():
            ring.zero_()  # slots that hold no token yet are compared too
        for b, n in enumerate(lens):
            k, v = _layer_kv(c, seed, layer, b, n)
            kvq.kvq_pack(cache, k[None], v[None], batch_begin=b)
        caches.append(cache)
    q, kn, vn = _token(c, seed)
    out = torch.empty(q.shape, dtype=torch.float32 if c["f32"] else torch.float16, device=DEV)
    n_splits = kvq.splits_for_lengths(cfg, [n + step for n in lens])
    ws = kvq.attn_workspace(cfg, n_splits, DEV)
    live = [x.seq_lens() for x in caches]
    start = [x.clone() for x in live]

    def work():
        for i, cache in enumerate(caches):
            if step:
                kvq.kvq_decode_step(cache, kn[i], vn[i], q[i], out=out[i], n_splits=n_splits,
                                    workspace=ws)
            else:
                kvq.kvq_decode_attn(cache, q[i], out=out[i], n_splits=n_splits, workspace=ws)
        if step:
            torch._foreach_copy_(live, start)

    result = {"out": out}
    graph = _capture(work)
    if step:
        # the updated cache: the new token in the windows, what it pushed out
        # of them in the pages
        for i, cache in enumerate(caches):
            if c["paged"]:
                result["pages%d" % i] = cache.pool
            elif min(nbs) > 0:
                result["pages%d" % i] = cache.pages()[:, :, :min(nbs)]
            result["k%d" % i], result["v%d" % i] = cache.resid()
            result["lens%d" % i] = cache.seq_lens()
    return dict(graph=graph, result=result, keep=(caches, q, kn, vn, ws, start))


def _chunks(c):
    return [min(c["chunk"], c["ctx"] - at) for at in range(0, c["ctx"], c["chunk"])]


def _prepare_prefill(c, seed):
    cfg = kvq.CacheConfig(batch=c["batch"], n_q_heads=c["hkv"], n_kv_heads=c["hkv"],
                          bits_k=c["bk"], bits_v=c["bv"], max_len=32 * (c["ctx"] // 32 + 16))
    cache = kvq.QuantKVCache(cfg, DEV)
    parts = []
    for i, n in enumerate(_chunks(c)):
        k = torch.empty(c["batch"], c["hkv"], n, D, dtype=torch.float16, device=DEV)
        v = torch.empty_like(k)
        for b in range(c["batch"]):
            k[b], v[b] = _layer_kv(c, seed, i, b, n)
        parts.append((k, v))
    k, v = cache.resid()
    k.zero_()
    v.zero_()
    return dict(cache=cache, parts=parts, result={
        "pages": cache.pages()[:, :, :kvq.packed_len(c["ctx"]) // G], "k": k, "v": v,
        "lens": cache.seq_lens()})


def _prepare_dgap(c, seed):
    head = kvq.DGAP(_dgap_weights(c, seed), K=c["k"], tau=c["tau"], device=DEV)
    fresh = _logits(c, seed)
    z = fresh.clone()
    ws = head.workspace(c["batch"], c["vocab"], DEV)
    outs = head.restore(z, workspace=ws)

    def work():
        z.copy_(fresh)
        head.restore(z, outputs=outs, workspace=ws)

    return dict(graph=_capture(work), result=dict(outs, logits=z), keep=(head, fresh, ws))


def prepare(case, seed):
    if case["kind"] in ("step", "attn"):
        return _prepare_decode(case, seed)
    if case["kind"] == "prefill":
        return _prepare_prefill(case, seed)
    if case["kind"] == "dgap":
        return _prepare_dgap(case, seed)
    zf, zq = _paired(case, seed)
    return dict(zf=zf, zq=zq, case=case)


def run(state):
    if "graph" in state:
        state["graph"].replay()
        return state["result"]
    if "parts" in state:
        cache = state["cache"]
        cache.reset()
        for k, v in state["parts"]:
            kvq.kvq_pack(cache, k, v)
        return state["result"]
    c = state["case"]
    o = kvq.drift_metrics(state["zf"], state["zq"], c["alpha"], c["window"], c["kmax"], 0.02, 0.5)
    kb, mean = kvq.drift_window(o["cov"], 0.6)
    return dict(o, k_b=kb, mean_cov=mean)


# ---------------------------------------------------------------------------
# Work and tolerance
# ---------------------------------------------------------------------------


def work(case):
    c = case
    if c["kind"] in ("step", "attn"):
        nbytes = flops = 0
        for n in _lengths(c):
            n += c["kind"] == "step"
            lq = kvq.packed_len(n)
            nbytes += c["hkv"] * (lq * (16 * (c["bk"] + c["bv"]) + 32) + (n - lq) * 4 * D)
            nbytes += c["hq"] * D * (6 if c["f32"] else 4)
            if c["kind"] == "step":
                nbytes += c["hkv"] * D * 4  # the token's ring slots
            flops += 4 * n * D * c["hq"]
        return dict(bytes=c["layers"] * nbytes, flops=c["layers"] * flops)
    if c["kind"] == "prefill":
        lq = kvq.packed_len(c["ctx"])
        rows = c["batch"] * c["hkv"]
        return dict(bytes=rows * (c["ctx"] * 4 * D + lq * (16 * (c["bk"] + c["bv"]) + 32)
                                  + min(160, c["ctx"]) * 4 * D),
                    flops=rows * 10 * c["ctx"] * D)
    if c["kind"] == "dgap":
        # the copy that brings the logits (read and write), their read by the
        # epilogue, and the weights
        nin = 5 * c["k"] + 8
        return dict(bytes=12 * c["batch"] * c["vocab"] + 4 * c["hidden"] * (nin + c["k"] + 10),
                    flops=c["batch"] * (8 * c["vocab"] + 2 * c["hidden"] * (nin + c["k"] + 9)))
    return dict(bytes=c["rows"] * (8 * c["vocab"] + 13 + 8 * c["kmax"]),
                flops=12 * c["rows"] * c["vocab"])


def tolerance(case):
    """About four times the distance from the 64-bit results that was seen:
    2.3e-4 for fp16 results (their own rounding) and one-bit values (fp16
    weights), 6e-5 for fp32 results (fp16 high and low parts, fp32 sums),
    7e-8 for the fp32 epilogue and the drift metrics (with room for the
    cancellation in small differences)."""
    if case["kind"] in ("step", "attn"):
        if case["f32"] and case["bv"] > 1:
            return {"rel": 2.5e-4, "max": 2.5e-3}
        return {"rel": 1e-3, "max": 6e-3}
    if case["kind"] == "prefill":
        return "exact"
    if case["kind"] == "dgap":
        return {"rel": 1e-6, "max": 1e-5}
    return {"rel": 1e-6, "max": 1e-5, "differ": 0.01}


# ---------------------------------------------------------------------------
# The same results in 64 bits, from the definitions
# ---------------------------------------------------------------------------


def _up32(x):
    """The least float32 not below x (float64)."""
    f = x.float()
    return torch.where(f.double() < x, torch.nextafter(f, torch.full_like(f, float("inf"))), f)


def _dequantized(x, bits, dim):
    """Groups of 32 along ``dim`` of x (fp16), quantized and read back."""
    levels = (1 << bits) - 1
    x = x.movedim(dim, -1)
    lo, hi = x.amin(-1).double(), x.amax(-1).double()
    span = _up32(hi - lo)
    s = _up32(span.double() / levels)
    s = torch.where(s.double() * levels < span.double(),
                    torch.nextafter(s, torch.full_like(s, float("inf"))), s)
    h = s.half()
    h = torch.where(h.double() < s.double(), (h.view(torch.int16) + 1).view(torch.float16), h)
    hf = h.float().unsqueeze(-1)
    ratio = (x.float() - lo.float().unsqueeze(-1)) / torch.where(hf > 0, hf, torch.ones_like(hf))
    code = torch.where(hf > 0, ratio.round().clamp(0, levels), torch.zeros_like(hf))
    return (lo.unsqueeze(-1) + h.double().unsqueeze(-1) * code.double()).movedim(-1, dim)


def _exact_attn(c, q, k, v):
    """softmax(q k^T / sqrt(d)) v of one sequence over its quantized cache:
    q [hq, d], k and v [hkv, n, d] fp16."""
    hkv, n, _ = k.shape
    lq = max(n - 128, 0) // G * G
    kh, vh = k.double(), v.double()
    if lq:
        kh[:, :lq] = _dequantized(k[:, :lq].reshape(hkv, lq // G, G, D), c["bk"], 2).reshape(
            hkv, lq, D)
        vh[:, :lq] = _dequantized(v[:, :lq].reshape(hkv, lq, D // G, G), c["bv"], 3).reshape(
            hkv, lq, D)
    p = torch.softmax(q.double().reshape(hkv, -1, D) @ kh.transpose(1, 2) / D ** 0.5, -1)
    return (p @ vh).reshape(-1, D)


def _exact_decode(c, seed):
    q, kn, vn = _token(c, seed)
    out = torch.empty(q.shape, dtype=torch.float64, device=DEV)
    for layer in range(c["layers"]):
        for b, n in enumerate(_lengths(c)):
            k, v = _layer_kv(c, seed, layer, b, n)
            if c["kind"] == "step":
                k = torch.cat([k, kn[layer, b].unsqueeze(1)], 1)
                v = torch.cat([v, vn[layer, b].unsqueeze(1)], 1)
            out[layer, b] = _exact_attn(c, q[layer, b], k, v)
    return {"out": out}


def _exact_dgap(c, seed):
    w = {k: v.double() for k, v in _dgap_weights(c, seed).items()}
    z = _logits(c, seed).double()
    k = c["k"]
    order = torch.sort(z, dim=-1, descending=True, stable=True)
    top, at = order.values[:, :k + 1], order.indices[:, :k]
    lse = torch.logsumexp(z, -1, keepdim=True)
    p = torch.exp(z - lse)
    win = top[:, :k]
    pw = torch.exp(win - lse)
    mass = pw.sum(-1)
    gaps = top[:, :-1] - top[:, 1:]
    qw = pw / mass.unsqueeze(-1)
    phi = torch.stack([-(p * (z - lse)).sum(-1), mass, pw[:, 0], gaps[:, 0],
                       (win[:, 0] - win[:, -1]) / (k - 1), gaps[:, :k - 1].amin(-1),
                       win.std(-1, correction=0), -(qw * qw.log()).sum(-1)], -1)
    f = torch.relu(phi @ w["det_w1"].T + w["det_b1"]) @ w["det_w2"] + w["det_b2"]
    risk = torch.sigmoid(f)
    rank = torch.arange(k, device=z.device, dtype=z.dtype).expand_as(win) / (k - 1)
    back = torch.cat([torch.zeros_like(win[:, :1]), gaps[:, :k - 1]], -1)
    xi = torch.stack([win - win[:, :1], win - lse, rank, back, gaps], -1).flatten(1)
    h = torch.relu(torch.cat([xi, phi], -1) @ w["cor_w1"].T + w["cor_b1"])
    delta = (h @ w["cor_w2"].T + w["cor_b2"]) * (risk > c["tau"]).unsqueeze(-1)
    return {"logits": z.scatter_add(1, at, delta), "topk_val": win + delta, "risk": risk,
            "features": phi, "topk_idx": None, "gate": None, "next_token": None}


def _exact_drift(c, seed):
    zf, zq = _paired(c, seed)
    outs = []
    for a, b in zip(zf.split(32), zq.split(32)):
        a, b = a.double(), b.double()
        pf, pq = torch.softmax(a, -1), torch.softmax(b, -1)
        fo = torch.sort(a, dim=-1, descending=True, stable=True).indices
        qo = torch.sort(b, dim=-1, descending=True, stable=True).indices[:, :c["kmax"]]
        alpha = float(torch.tensor(c["alpha"], dtype=torch.float32))
        m = (torch.cumsum(pf.gather(1, fo), -1) < alpha).sum(-1) + 1
        first = torch.arange(a.shape[1], device=a.device) < m.unsqueeze(-1)
        in_c = torch.zeros_like(first).scatter(1, fo, first)
        in_s = torch.zeros_like(in_c).scatter(1, qo[:, :c["window"]], True)
        u = in_c | in_s
        x, y = pf * u, pq * u
        d = (x / x.sum(-1, keepdim=True) - y / y.sum(-1, keepdim=True)).norm(dim=-1)
        cov = torch.cumsum((pf * in_c).gather(1, qo), -1)
        outs.append(((pf * (in_c & in_s)).sum(-1), d, cov))
    ct, d, cov = (torch.cat(x) for x in zip(*outs))
    return {"c_t": ct, "d_loc": d, "cov": cov, "mean_cov": cov.mean(0), "m_t": None, "y_t": None,
            "k_b": None}


def exact(case, seed):
    if case["kind"] in ("step", "attn"):
        return _exact_decode(case, seed)
    if case["kind"] == "dgap":
        return _exact_dgap(case, seed)
    if case["kind"] == "drift":
        return _exact_drift(case, seed)
    return None  # codes and copies: whole values
