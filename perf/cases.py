"""What a user of the library has it do, as cases that can be timed and compared.

Five kinds of pass, each through the public calls of paper_2609_33135_b200.binding with buffers that a serving program
keeps between calls:

  prefill      a whole prompt from BF16 Q, K, V: stage 1 (statistics, NVFP4 Q and K, Delta_S, FP8 V), then attention
  quantize     stage 1 alone (the encoder side: operands for a later attention call)
  cache_write  one request's prompt quantized into the pages of the decode cache
  chunk        chunked prefill: a chunk of queries per request, its K and V appended to the pages with the frozen
               statistics, then attention over the pages
  decode       one serving step of a batch: append the new token's K and V, quantize the query, split-KV decode

Shapes are those of the library's workloads, tests and benchmark (GQA 32:8 and 40:8, head_dim 128, 256 to 131072 tokens,
64-token pages) and generic ones between them.  Values follow the workloads' recipe: N(0, 1) with per-channel offsets and
outlier channels on K, optionally offsets on Q.
"""
import math
import random

import torch

from paper_2609_33135_b200 import binding, workloads

D = 128
PAGE = 64


def _prefill(name, B, N, H_q, H_kv, causal=True, N_q=0, smooth=True, q_bias=False, v_scale=1.0):
    return {"name": name, "kind": "prefill", "B": B, "N": N, "N_q": N_q or N, "H_q": H_q, "H_kv": H_kv, "causal": causal,
            "smooth": smooth, "q_bias": q_bias, "v_scale": v_scale}


def listed():
    return [
        # the smallest call: one head of 256 tokens, all launches and host work
        _prefill("prefill_tiny", 1, 256, 1, 1, causal=False),
        # several short prompts of a small GQA model at once, ragged length
        _prefill("prefill_short_batch", 4, 777, 8, 2, q_bias=True),
        # non-causal multi-head attention over short sequences (an encoder), ragged last tile
        _prefill("encoder_batch", 8, 577, 16, 16, causal=False),
        # an ordinary chat prompt on the 40:8 shape, ragged
        _prefill("prefill_2k", 1, 1999, 40, 8, q_bias=True),
        # the benchmark's long prompt
        _prefill("prefill_16k", 1, 16384, 32, 8),
        # the longest context of the benchmark: the largest case
        _prefill("prefill_128k", 1, 131072, 32, 8),
        # stage 1 alone at the 40:8 shape, where it runs at memory speed
        dict(_prefill("quantize_32k", 1, 32768, 40, 8, q_bias=True), kind="quantize"),
        # a new request's prompt written to the cache, ragged last page
        {"name": "cache_write_9k", "kind": "cache_write", "N": 9001, "H_q": 32, "H_kv": 8, "smooth": True, "v_scale": 1.0},
        # a step of chunked prefill: four requests, 512 new tokens each on ragged contexts
        {"name": "chunk_512", "kind": "chunk", "B": 4, "N_q": 512, "len_lo": 2000, "len_hi": 16000, "H_q": 32, "H_kv": 8,
         "smooth": True, "v_scale": 1.0},
        # interactive decoding of one request with a middling context: latency
        {"name": "decode_single", "kind": "decode", "B": 1, "len_lo": 4097, "len_hi": 4097, "H_q": 32, "H_kv": 8,
         "smooth": True, "v_scale": 1.0},
        # a chat server's decode batch: many requests, short ragged contexts
        {"name": "decode_batch", "kind": "decode", "B": 64, "len_lo": 100, "len_hi": 4000, "H_q": 40, "H_kv": 8,
         "smooth": True, "v_scale": 1.0},
        # the benchmark's decode batch: 32 long contexts, bound by reading the cache
        {"name": "decode_long", "kind": "decode", "B": 32, "len_lo": 16384, "len_hi": 131072, "H_q": 32, "H_kv": 8,
         "smooth": True, "v_scale": 1.0},
    ]


def _log_int(rng, lo, hi):
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def _tokens(rng, lo, hi):
    n, r = _log_int(rng, lo, hi), rng.random()
    if r < 0.25:      # a whole number of 128-token tiles, as padded batches have
        n = max(128, n // 128 * 128)
    elif r < 0.5:     # just past one or short of it
        n = max(128, n // 128 * 128) + rng.choice((-1, 1))
    return max(lo, min(hi, n))


def draw(rng):
    """Another case of the ranges above: prompts of 64 to 131072 tokens, contexts of 1 to 131072, every GQA group of the listed
    shapes and of the tests, with and without smoothing, causal and not, more keys than queries."""
    H_q, H_kv = rng.choice(((1, 1), (4, 4), (8, 2), (8, 1), (16, 16), (32, 8), (32, 8), (40, 8), (40, 8)))
    smooth = rng.random() < 0.85
    v_scale = rng.choice((1.0, 1.0, 0.5))
    kind = rng.choice(("prefill", "prefill", "prefill", "quantize", "cache_write", "chunk", "decode", "decode"))
    if kind in ("prefill", "quantize"):
        causal = rng.random() < 0.75
        while True:
            N, B = _tokens(rng, 64, 131072), _log_int(rng, 1, 16)
            N_q = N if rng.random() < 0.8 else _tokens(rng, 1, N)
            c = dict(_prefill("", B, N, H_q, H_kv, causal, N_q, smooth, rng.random() < 0.5, v_scale), kind=kind)
            if B * max(N, N_q) * H_q <= 131072 * 32 and work(c)["flops"] <= _largest():
                break
    elif kind == "cache_write":
        c = {"kind": kind, "N": _tokens(rng, 64, 65536), "H_q": H_q, "H_kv": H_kv, "smooth": smooth, "v_scale": v_scale}
    elif kind == "chunk":
        while True:
            B, N_q, hi = _log_int(rng, 1, 8), _tokens(rng, 64, 4096), _tokens(rng, 256, 65536)
            if N_q < hi and B * hi <= 131072:
                break
        c = {"kind": kind, "B": B, "N_q": N_q, "len_lo": _log_int(rng, N_q + 1, hi), "len_hi": hi, "H_q": H_q, "H_kv": H_kv,
             "smooth": smooth, "v_scale": v_scale}
    else:
        while True:
            B, hi = _log_int(rng, 1, 256), _tokens(rng, 16, 131072)
            if B * hi <= 1 << 21:
                break
        c = {"kind": kind, "B": B, "len_lo": _log_int(rng, 1, hi), "len_hi": hi, "H_q": H_q, "H_kv": H_kv, "smooth": smooth,
             "v_scale": v_scale}
    c.pop("name", None)
    return c


def _largest():
    return max(work(c)["flops"] for c in listed())


def _lengths(case):
    """Context lengths of a batch: a function of the case, so that its work is."""
    r = random.Random("%d %d %d" % (case["B"], case["len_lo"], case["len_hi"]))
    return [r.randint(case["len_lo"], case["len_hi"]) for _ in range(case["B"])]


def _visible_pairs(N_q, N_kv, causal):
    if not causal:
        return N_q * N_kv
    hidden = min(N_q, N_kv) - 1   # bottom-right aligned: query i sees keys 0 .. i + N_kv - N_q
    if N_q <= N_kv:
        return N_q * N_kv - hidden * (hidden + 1) // 2
    return N_kv * (N_kv + 1) // 2


def work(case):
    H_q, H_kv, kind = case["H_q"], case["H_kv"], case["kind"]
    cached = H_kv * (64 + 8 + D) + (2 * H_q if case["smooth"] else 0)   # bytes of one token in the cache
    if kind in ("prefill", "quantize"):
        B, N, N_q = case["B"], case["N"], case["N_q"]
        read = 2 * D * B * (N_q * H_q + 2 * N * H_kv)
        if kind == "quantize":
            return {"bytes": read + B * (N_q * H_q * 72 + N * cached), "flops": 0}
        return {"bytes": read + 2 * D * B * N_q * H_q, "flops": 4 * D * B * H_q * _visible_pairs(N_q, N, case["causal"])}
    if kind == "cache_write":
        return {"bytes": case["N"] * (4 * D * H_kv + cached), "flops": 0}
    lens = _lengths(case)
    n = case["N_q"] if kind == "chunk" else 1
    new = case["B"] * n * (4 * D * H_q + 4 * D * H_kv + cached)   # queries, outputs, new keys and values, their cache bytes
    return {"bytes": sum(lens) * cached + new, "flops": 4 * D * H_q * sum(_visible_pairs(n, L, True) for L in lens)}


def tolerance(case):
    """Stage 1 is specified to the bit.  Attention outputs are BF16 from FP32 accumulation: the two work arrangements of the
    prefill kernel, which rescale and add in different orders, differ by 2e-5 to 1.3e-4 (relative 2-norm over the listed
    cases) and by one BF16 step at most; a probability that lies on a rounding boundary of its 8-bit code may move one short
    row by up to 6 %."""
    if case["kind"] in ("quantize", "cache_write"):
        return "exact"
    return {"rel": 5e-4, "max": 0.06}


def _flags(case):
    return binding.MPFA_SMOOTH if case["smooth"] else 0


class _Draws:
    """Seeded inputs on the GPU: offsets and outlier channels on K, offsets on Q."""

    def __init__(self, case, seed):
        self.g = torch.Generator(device="cuda")
        self.g.manual_seed(seed)
        H_kv = case["H_kv"]
        self.bias, self.factor = (t.cuda() for t in workloads.k_structure(seed, H_kv, max(1, round(0.01 * H_kv * D))))
        self.q_off = torch.randn(case["H_q"], D, generator=self.g, device="cuda")

    def normal(self, *shape):
        return torch.randn(*shape, generator=self.g, device="cuda")

    def q(self, *tokens):
        return self.normal(*tokens, *self.q_off.shape).add_(self.q_off).bfloat16()

    def k(self, *tokens):
        return self.normal(*tokens, *self.bias.shape).mul_(self.factor).add_(self.bias).bfloat16()

    def v(self, *tokens):
        return self.normal(*tokens, *self.bias.shape).bfloat16()


def _paged_cache(case, d, lens):
    """An empty cache with shuffled pages for requests of these lengths, and the frozen query statistics of each request."""
    B, H_q, H_kv = len(lens), case["H_q"], case["H_kv"]
    pages = [-(-L // PAGE) for L in lens]
    order = torch.randperm(sum(pages) + 3, generator=d.g, device="cuda").to(torch.int32)
    table = torch.full((B, max(pages)), -1, dtype=torch.int32, device="cuda")
    at = 0
    for b, n in enumerate(pages):
        table[b, :n] = order[at:at + n]
        at += n
    kv = binding.PagedKV.empty(sum(pages) + 3, H_q, H_kv, with_delta=case["smooth"])
    stats = binding.Stats.empty(B, H_q, H_kv)
    ws = binding.quantize_workspace(B, H_q, H_kv)
    binding.mpfa_quantize_qk(d.q(B, 256), None, _flags(case), stats, binding.Fp4Tensor.empty(B, H_q, 256), None, None, ws)
    return {"kv": kv, "table": table, "stats": stats, "ws": ws}


def prepare(case, seed):
    kind, H_q, H_kv = case["kind"], case["H_q"], case["H_kv"]
    st = {"case": case, "kind": kind, "scale": 1.0 / math.sqrt(D), "flags": _flags(case), "v_scale": case["v_scale"]}
    if kind in ("prefill", "quantize"):
        B, N, N_q = case["B"], case["N"], case["N_q"]
        q, k, v = workloads.make_qkv(seed, B, N_q, N, H_q, H_kv, q_bias=case["q_bias"], device="cuda")
        ws = binding.quantize_workspace(B, H_q, H_kv)
        s1 = binding.stage1(q, k, v, case["smooth"], case["v_scale"], ws)   # allocates the operand buffers that are kept
        st.update(q=q, k=k, v=v, ws=ws, s1=s1)
        if kind == "prefill":
            st.update(out=torch.empty(B, N_q, H_q, D, dtype=torch.bfloat16, device="cuda"),
                      status=torch.zeros(1, dtype=torch.int32, device="cuda"))
        return st
    d = _Draws(case, seed)
    if kind == "cache_write":
        st.update(_paged_cache(case, d, [case["N"]]), k=d.k(case["N"]), v=d.v(case["N"]))
        return st
    lens, n = _lengths(case), case["N_q"] if kind == "chunk" else 1
    B = len(lens)
    st.update(_paged_cache(case, d, lens))
    for b, L in enumerate(lens):   # what the requests already hold
        n_old = max(1, L - n)
        binding.mpfa_quantize_kv_paged(d.k(n_old), d.v(n_old), 0, H_q, st["flags"], st["stats"].request(b), st["v_scale"], st["kv"],
                                       st["table"][b], st["ws"])
    st.update(q=d.q(B, n), k=d.k(B, n), v=d.v(B, n), q4=binding.Fp4Tensor.empty(B, H_q, n),
              lens=torch.tensor(lens, dtype=torch.int32, device="cuda"),
              out=torch.empty(B, n, H_q, D, dtype=torch.bfloat16, device="cuda"),
              status=torch.zeros(1, dtype=torch.int32, device="cuda"))
    if kind == "chunk":
        st["per_request"] = [(st["k"][b], st["v"][b], L - n, st["stats"].request(b), st["table"][b]) for b, L in enumerate(lens)]
    else:
        st["positions"] = st["lens"] - 1
        st["ws"] = binding.decode_workspace(B, H_q, H_kv, st["table"].shape[1])
    return st


def _cache(kv):
    return [kv.k_codes, kv.k_sf, kv.v_fp8] + ([] if kv.delta is None else [kv.delta])


def run(st):
    kind, H_q = st["kind"], st["case"]["H_q"]
    if kind in ("prefill", "quantize"):
        s1 = binding.stage1(st["q"], st["k"], st["v"], st["case"]["smooth"], st["v_scale"], st["ws"], st["s1"])
        if kind == "quantize":
            x = s1.stats
            return [s1.q.codes, s1.q.sf, s1.k.codes, s1.k.sf, s1.v_fp8, s1.delta, x.q_mean, x.k_mean, x.q_gscale, x.k_gscale]
        out, _, status = binding.prefill(s1, st["case"]["causal"], st["scale"], out=st["out"], status=st["status"])
        return [out, status]
    kv, stats = st["kv"], st["stats"]
    if kind == "cache_write":
        binding.mpfa_quantize_kv_paged(st["k"], st["v"], 0, H_q, st["flags"], stats, st["v_scale"], kv, st["table"][0], st["ws"])
        return _cache(kv) + [stats.k_mean, stats.k_gscale]
    frozen = st["flags"] | binding.MPFA_STATS_FROZEN
    if kind == "chunk":
        for k, v, first, request, row in st["per_request"]:
            binding.mpfa_quantize_kv_paged(k, v, first, H_q, frozen, request, st["v_scale"], kv, row, None)
        binding.mpfa_quantize_qk(st["q"], None, frozen, stats, st["q4"], None, None, None)
        binding.mpfa_prefill_paged(st["q4"], kv, st["table"], st["lens"], stats, st["v_scale"], st["scale"], st["out"], None,
                                   st["status"])
    else:
        binding.mpfa_append_kv_paged(st["k"], st["v"], H_q, st["flags"], stats, st["v_scale"], kv, st["table"], st["positions"])
        binding.mpfa_quantize_qk(st["q"], None, frozen, stats, st["q4"], None, None, None)
        binding.mpfa_decode(st["q4"], kv, st["table"], st["lens"], stats, st["v_scale"], st["scale"], st["out"], None, st["ws"],
                            st["status"])
    return [st["out"], st["status"]] + _cache(kv)
