"""The work that the framework's performance is measured on: what a serving program has it do, through the public
entry points of ``api`` and ``decode_api``, from the smallest calls to the largest configuration of ``workloads``.

A case is a dict of plain values.  ``kind`` says which path it takes:

  prefill   one call of ``hybrid_prefill``: select the vertical keys, quantize Q, K and V, hybrid attention
  mass      the same three stages called one by one, with the column-mass selector (Eq. 4-5) in the first
  chunk     chunked prefill: the last ``Lq`` rows of a context of ``L`` keys (Algorithm 2's query block), with LSE
  varlen    a ragged batch of prompts through ``hybrid_prefill_varlen``
  freeze    Algorithm 4: the prefill cache turned into the hybrid decode cache
  decode    one decode step: append the token's K and V rows, then Algorithm 3's attention
  ragged    the same step for a batch of sequences of different lengths
"""
import math
import random

import torch

from paper_2608_27875_b200 import api, decode_api, workloads

D = 128
FORMATS = {"int8": (workloads.FMT_INT8,) * 3, "fp8": (workloads.FMT_FP8_E4M3,) * 3,
           "int4": (workloads.FMT_INT4, workloads.FMT_INT4, workloads.FMT_FP8_E4M3)}
CACHE_FORMATS = {"int4": workloads.FMT_INT4, "int8": workloads.FMT_INT8, "fp8": workloads.FMT_FP8_E4M3}
OUT = {"fp32": torch.float32, "bf16": torch.bfloat16}
CODE_BYTES = {workloads.FMT_INT8: 1.0, workloads.FMT_FP8_E4M3: 1.0, workloads.FMT_INT4: 0.5}


def _prefill(name, cfg, fmt, out):
    w = workloads.CONFIGS[cfg]
    return dict(name=name, kind="prefill", B=w.B, Hq=w.Hq, Hkv=w.Hkv, L=w.L, window=w.window, k=w.k, fmt=fmt, out=out,
                outliers=w.outlier_channels)


def listed():
    return [
        # a short prompt on two heads: a model's head shard, or a first request; launches and latency are what it costs
        _prefill("prefill_2k", "c0", "int8", "fp32"),
        # an ordinary prompt on one layer of a 32/8-head model
        _prefill("prefill_8k", "c1", "int8", "fp32"),
        # the benchmark's default: a long document at the lowest bit widths
        _prefill("prefill_32k", "c2", "int4", "fp32"),
        # the longest context of the configurations
        _prefill("prefill_128k", "c3", "int8", "fp32"),
        # four prompts of one length, outlier channels in K, output in the model's own type
        _prefill("prefill_16k_b4", "c4", "int8", "bf16"),
        # the paper's own definition of the vertical score, on a prompt whose length fills neither a block nor a tile
        dict(name="prefill_mass", kind="mass", B=1, Hq=32, Hkv=8, L=12007, window=512, k=241, fmt="fp8", out="bf16",
             block=64, n_queries=16),
        # chunked prefill late in a long context
        dict(name="chunk_1k", kind="chunk", B=1, Hq=32, Hkv=8, L=32768, Lq=1024, window=1024, k=656, fmt="int4", out="bf16",
             block=64),
        # continuous batching: prompts of different lengths arrive together
        dict(name="varlen_8", kind="varlen", n_seq=8, Hq=32, Hkv=8, lo=130, hi=6000, window=256, pct=2, fmt="int8", out="bf16",
             lengths=17),
        # the end of the prefill of a batch of long prompts: the decode cache is built
        dict(name="freeze_b8", kind="freeze", B=8, Hq=32, Hkv=8, L=32768, window=1024, k=656, fmt="int4", group=64),
        # interactive decoding, one sequence
        dict(name="decode_b1", kind="decode", B=1, Hq=32, Hkv=8, L=8192, window=512, k=164, fmt="int4", group=64, staged=37,
             out="bf16"),
        # batched decoding of long contexts
        dict(name="decode_b8", kind="decode", B=8, Hq=32, Hkv=8, L=32768, window=1024, k=656, fmt="int4", group=64, staged=100,
             out="bf16"),
        # a serving batch: sequences of different lengths, one token each
        dict(name="ragged_16", kind="ragged", n_seq=16, Hq=32, Hkv=8, lo=600, hi=24000, window=512, pct=2, lengths=5,
             out="bf16"),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _pct(n, p):
    return -(-n * p // 100)


def draw(rng: random.Random):
    kind = rng.choice(["prefill", "prefill", "mass", "chunk", "varlen", "freeze", "decode", "decode", "ragged"])
    Hq, Hkv = rng.choice([(2, 2), (8, 8), (16, 4), (32, 8), (32, 8), (40, 8), (32, 4)])
    fmt, out = rng.choice(["int8", "fp8", "int4"]), rng.choice(["fp32", "bf16"])
    if kind == "prefill":
        B, L = rng.choice([1, 1, 2, 4]), _log(rng, 200, 131072)
        while B * Hq * L * L > 32 * 131072 ** 2 // 2:
            L //= 2
        W = rng.choice([64, 128, 512, 1024])
        return dict(kind=kind, B=B, Hq=Hq, Hkv=Hkv, L=L, window=W, k=_pct(max(0, L - W), rng.choice([1, 2, 3])), fmt=fmt, out=out,
                    outliers=rng.random() < 0.25)
    if kind == "mass":
        L, W = _log(rng, 1500, 24000), rng.choice([128, 512, 1024])
        return dict(kind=kind, B=1, Hq=Hq, Hkv=Hkv, L=L, window=W, k=_pct(L - W, 2), fmt=fmt, out=out,
                    block=rng.choice([32, 64, 64, 128]), n_queries=rng.choice([4, 8, 16, 30, 64]))
    if kind == "chunk":
        L = _log(rng, 4096, 65536)
        W = rng.choice([128, 512, 1024])
        return dict(kind=kind, B=rng.choice([1, 1, 2]), Hq=Hq, Hkv=Hkv, L=L, Lq=_log(rng, 64, min(4096, L)), window=W,
                    k=_pct(L - W, 2), fmt=fmt, out=out, block=rng.choice([64, 64, 64, 32, 128]))
    if kind == "varlen":
        lo = _log(rng, 40, 1000)
        return dict(kind=kind, n_seq=rng.randint(2, 8), Hq=Hq, Hkv=Hkv, lo=lo, hi=_log(rng, 2 * lo, 12000),
                    window=rng.choice([64, 256, 512]), pct=rng.choice([1, 2, 3]), fmt=fmt, out=out, lengths=rng.randint(0, 999))
    if kind == "freeze":
        B, L, W = rng.randint(1, 8), _log(rng, 700, 32768), rng.choice([128, 512, 1024])
        W = min(W, L // 2)
        return dict(kind=kind, B=B, Hq=Hq, Hkv=Hkv, L=L, window=W, k=_pct(L - W, 2), fmt=fmt, group=rng.choice([32, 64, 64, 128]))
    if kind == "decode":
        B, L, W = rng.choice([1, 1, 2, 4, 8, 16]), _log(rng, 700, 65536), rng.choice([128, 512, 1024])
        while B * L > 16 * 32768:
            L //= 2
        W = min(W, L // 2)
        return dict(kind=kind, B=B, Hq=Hq, Hkv=Hkv, L=L, window=W, k=_pct(L - W, 2), fmt=fmt, group=rng.choice([32, 64, 64, 128]),
                    staged=rng.randint(0, 120), out=out)
    lo = _log(rng, 100, 4000)
    return dict(kind="ragged", n_seq=rng.randint(2, 32), Hq=Hq, Hkv=Hkv, lo=lo, hi=_log(rng, 2 * lo, 24000),
                window=rng.choice([128, 512]), pct=2, lengths=rng.randint(0, 999), out=out)


# ---- inputs ---------------------------------------------------------------------------------------------------------
def _lengths(case):
    """The batch's lengths: spread over their logarithm, fixed by the case (a batch's shape is not the inputs' values)."""
    r = random.Random(case["lengths"])
    return [_log(r, case["lo"], case["hi"]) for _ in range(case["n_seq"])]


def _k_of(case, n):
    return _pct(max(0, n - case["window"]), case["pct"])


def _qkv(g, B, Hq, Hkv, L, Lq=None, outliers=False):
    """bf16 Q, K, V as ``workloads`` draws them: normal values, persistent vertical lines - one direction per KV head that
    L / 128 planted keys (the first among them) and every query carry - and, where asked for, four outlier channels."""
    dev = "cuda"
    u = torch.randn(B, Hkv, 1, D, generator=g, device=dev)
    u = u / u.norm(dim=-1, keepdim=True)
    k = torch.randn(B, Hkv, L, D, generator=g, device=dev)
    if outliers:
        k[..., list(workloads.OUTLIER_CHANNELS)] *= 20.0
    n = max(1, L // 128)
    pos = torch.rand(B, Hkv, L, generator=g, device=dev).topk(n, dim=-1).indices
    pos[..., 0] = 0
    k.scatter_add_(2, pos.unsqueeze(-1).expand(-1, -1, -1, D), (4.0 * u).expand(-1, -1, n, -1))
    k = k.bfloat16()
    v = torch.randn(B, Hkv, L, D, generator=g, device=dev).bfloat16()
    q = torch.randn(B, Hq, Lq or L, D, generator=g, device=dev)
    q += (1.5 * u).repeat_interleave(Hq // Hkv, dim=1)
    return q.bfloat16(), k, v


def _rows(g, *shape):
    return torch.randn(*shape, generator=g, device="cuda").bfloat16()


class State:
    def __init__(self, case, **kw):
        self.case = case
        self.__dict__.update(kw)


def prepare(case, seed):
    g = torch.Generator(device="cuda").manual_seed(seed)
    kind, Hq, Hkv = case["kind"], case["Hq"], case["Hkv"]
    if kind in ("prefill", "mass"):
        q, k, v = _qkv(g, case["B"], Hq, Hkv, case["L"], outliers=case.get("outliers", False))
        return State(case, q=q, k=k, v=v)
    if kind == "chunk":
        q, k, v = _qkv(g, case["B"], Hq, Hkv, case["L"], Lq=case["Lq"])
        return State(case, q=q, k=k, v=v)
    if kind == "varlen":
        seqs = [_qkv(g, 1, Hq, Hkv, n) for n in _lengths(case)]
        qs, ks, vs = ([s[i][0] for s in seqs] for i in range(3))
        return State(case, qs=qs, ks=ks, vs=vs, k_per_seq=[_k_of(case, n) for n in _lengths(case)])
    if kind in ("freeze", "decode"):
        B, L, W, kk, fmt = case["B"], case["L"], case["window"], case["k"], CACHE_FORMATS[case["fmt"]]
        q, k, v = _qkv(g, B, Hq, Hkv, L, Lq=min(W, L))
        idx = api.hyq_select_vertical(q[:, ::Hq // Hkv].contiguous(), k, W, kk)      # one set per KV head
        desc = decode_api.make_desc(B, Hq, Hkv, L, W, kk, 128, group=case["group"], fmt=fmt)
        cache = decode_api.alloc_cache(desc)
        if kind == "freeze":
            return State(case, k=k, v=v, idx=idx, cache=cache)
        decode_api.hyq_freeze(k, v, idx, W, Hq, cache=cache, group=case["group"], fmt=fmt)
        for name in ("k_s", "v_s"):
            cache.buffers[name].zero_()
            cache.buffers[name][:, :, :case["staged"]] = _rows(g, B, Hkv, case["staged"], D)
        desc.n_staging = case["staged"] + 1
        ws = torch.empty(max(16, decode_api.hyq_hybrid_attention_decode_workspace(cache)), dtype=torch.uint8, device="cuda")
        return State(case, q=q[:, :, -1].contiguous(), cache=cache, k_new=_rows(g, B, Hkv, D), v_new=_rows(g, B, Hkv, D), ws=ws,
                     out=torch.empty(B, Hq, D, dtype=OUT[case["out"]], device="cuda"))
    ns, W = _lengths(case), case["window"]
    B = len(ns)
    cache = decode_api.RaggedKvCache(B, Hq, Hkv, max(ns), W, max(_k_of(case, n) for n in ns))
    staged = [(7 * b + n) % 100 for b, n in enumerate(ns)]
    for name in ("k_s", "v_s"):
        cache.batch.buffers[name].zero_()
    q_t = []
    for b, n in enumerate(ns):
        q, k, v = _qkv(g, 1, Hq, Hkv, n, Lq=min(W, n))
        kk = _k_of(case, n)
        idx = api.hyq_select_vertical(q[:, ::Hq // Hkv].contiguous(), k, W, kk) if kk else None
        cache.freeze_sequence(b, k, v, idx)
        for name in ("k_s", "v_s"):
            cache.batch.buffers[name][b, :, :staged[b]] = _rows(g, Hkv, staged[b], D)
        q_t.append(q[0, :, -1])
    ws = torch.empty(max(16, decode_api.hyq_hybrid_attention_decode_workspace(cache.batch)), dtype=torch.uint8, device="cuda")
    return State(case, cache=cache, q=torch.stack(q_t), staged=torch.tensor(staged, dtype=torch.int32), ws=ws,
                 k_new=_rows(g, B, Hkv, D), v_new=_rows(g, B, Hkv, D),
                 out=torch.empty(B, Hq, D, dtype=OUT[case["out"]], device="cuda"))


# ---- one pass -------------------------------------------------------------------------------------------------------
def run(s):
    case = s.case
    kind = case["kind"]
    if kind == "prefill":
        return api.hybrid_prefill(s.q, s.k, s.v, case["window"], case["k"], FORMATS[case["fmt"]], out_dtype=OUT[case["out"]])
    if kind in ("mass", "chunk"):
        fmts, W, bt = FORMATS[case["fmt"]], case["window"], case["block"]
        if kind == "mass":
            idx = api.hyq_select_vertical_mass(s.q, s.k, W, case["k"], n_queries=case["n_queries"])
            lse = None
        else:
            idx = api.hyq_select_vertical(s.q, s.k, W, case["k"])
            lse = torch.empty(s.q.shape[:3], dtype=torch.float32, device=s.q.device)
        qc, qs = api.hyq_quantize_blocks(s.q, fmts[0], bt)
        kc, ks = api.hyq_quantize_blocks(s.k, fmts[1], bt)
        vc, vs = api.hyq_quantize_blocks(s.v, fmts[2], bt)
        out = api.hyq_hybrid_attention_prefill(s.q, s.k, s.v, qc, kc, vc, qs, ks, vs, fmts, idx, W, out_dtype=OUT[case["out"]],
                                               lse=lse, block_tokens=bt)
        return dict(idx=idx, q_codes=qc, k_codes=kc, v_codes=vc, q_scales=qs, k_scales=ks, v_scales=vs, out=out, lse=lse)
    if kind == "varlen":
        return api.hybrid_prefill_varlen(s.qs, s.ks, s.vs, case["window"], s.k_per_seq, FORMATS[case["fmt"]],
                                         out_dtype=OUT[case["out"]])
    if kind == "freeze":
        decode_api.hyq_freeze(s.k, s.v, s.idx, case["window"], case["Hq"], cache=s.cache, group=case["group"],
                              fmt=CACHE_FORMATS[case["fmt"]])
        nq = int(s.cache.sizes.quantized_rows)
        buf = dict(s.cache.buffers)
        buf.pop("k_s"), buf.pop("v_s")
        buf["kq_codes"] = buf["kq_codes"][:, :, :nq]
        buf["vq_codes"] = buf["vq_codes"][:, :, :nq // 16]       # whole tiles (padding rows are unspecified)
        return buf
    if kind == "decode":
        s.cache.desc.n_staging = case["staged"]                  # the step of the state, however often it is taken
        s.cache.append(s.k_new, s.v_new)
        decode_api.hyq_hybrid_attention_decode(s.q, s.cache, out=s.out, workspace=s.ws)
        return dict(out=s.out, k_s=s.cache.buffers["k_s"], v_s=s.cache.buffers["v_s"])
    s.cache.lengths_host[:, 3] = s.staged
    for b in range(case["n_seq"]):
        s.cache.append(b, s.k_new[b], s.v_new[b])
    decode_api.hyq_hybrid_attention_decode_ragged(s.q, s.cache, out=s.out, workspace=s.ws)
    return dict(out=s.out, k_s=s.cache.batch.buffers["k_s"], v_s=s.cache.batch.buffers["v_s"], lengths=s.cache.lengths)


# ---- what a pass cannot do without ----------------------------------------------------------------------------------
def _prefill_work(B, Hq, Hkv, L, Lq, k, fmts, out, block=64):
    q, kv = B * Hq * Lq * D, B * Hkv * L * D
    byts = 2 * (q + 2 * kv) + q * CODE_BYTES[fmts[0]] + kv * (CODE_BYTES[fmts[1]] + CODE_BYTES[fmts[2]])
    byts += 4 * (B * Hq * -(-Lq // block) + 2 * B * Hkv * -(-L // block)) + 4 * B * Hq * k + q * (4 if out == "fp32" else 2)
    pairs = B * Hq * (Lq * (L - Lq) + Lq * (Lq + 1) // 2)
    return byts, 4 * D * pairs


def _cache_bytes(heads, nq, rows, fmt, group):
    code = 1.0 if CACHE_FORMATS[fmt] == workloads.FMT_INT4 else 2.0             # K and V of one channel
    return heads * (nq * D * code + 8 * -(-nq // group) + 4 * D * rows)


def work(case):
    kind, Hq, Hkv = case["kind"], case["Hq"], case["Hkv"]
    if kind in ("prefill", "mass", "chunk"):
        B, L = case["B"], case["L"]
        byts, flops = _prefill_work(B, Hq, Hkv, L, case.get("Lq", L), case["k"], FORMATS[case["fmt"]], case["out"], case.get("block", 64))
        if kind == "mass":
            flops += 2 * D * B * Hq * case["n_queries"] * L                    # the tail queries' scores
        return dict(bytes=byts, flops=flops)
    if kind == "varlen":
        ws = [_prefill_work(1, Hq, Hkv, n, n, _k_of(case, n), FORMATS[case["fmt"]], case["out"]) for n in _lengths(case)]
        return dict(bytes=sum(w[0] for w in ws), flops=sum(w[1] for w in ws))
    if kind in ("freeze", "decode"):
        B, L, W, kk = case["B"], case["L"], min(case["window"], case["L"]), case["k"]
        heads, nq = B * Hkv, L - W - kk
        if kind == "freeze":
            return dict(bytes=heads * L * D * 4 + _cache_bytes(heads, nq, kk + W, case["fmt"], case["group"]), flops=0)
        rows = kk + W + case["staged"] + 1
        return dict(bytes=_cache_bytes(heads, nq, rows, case["fmt"], case["group"]) + 4 * B * Hq * D, flops=4 * D * B * Hq * (nq + rows))
    byts = flops = 0
    for b, n in enumerate(_lengths(case)):
        W, kk = min(case["window"], n), _k_of(case, n)
        nq, rows = n - W - kk, kk + W + (7 * b + n) % 100 + 1
        byts += _cache_bytes(Hkv, nq, rows, "int4", 64) + 4 * Hq * D
        flops += 4 * D * Hq * (nq + rows)
    return dict(bytes=byts, flops=flops)


def tolerance(case):
    # Index sets, codes, scales and copied rows stay the same bit for bit.  The attention's weights enter the value
    # product in 16 bits and its output may be stored as bf16.  Measured on these inputs, the tensor-core prefill against
    # the fp32 CUDA-core kernel and the decode attention against itself with other slices: 2.8e-4 (largest difference
    # 4.2e-3) for fp32 outputs, 1.06e-3 (7.8e-3, one step of bf16) for bf16 ones; four times that is allowed.
    if case["kind"] == "freeze":
        return "exact"
    return {"rel": 1.2e-3, "max": 1.7e-2} if case["out"] == "fp32" else {"rel": 4e-3, "max": 3.1e-2}
