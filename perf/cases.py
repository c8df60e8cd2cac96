"""Performance cases of the novakv library: what a serving engine calls it for, through its public classes.

One case is one pass of one attention layer: a decode step (append this step's tokens, then attend over the index
cache), the encoding of a prompt chunk, a sliding-window layer on the BF16 cache, or the host-buffer step.  Sizes are
those of this repository's workloads and of its benchmark sweep; ``draw`` gives others of the same ranges.

    listed() -> cases        draw(rng) -> case        prepare(case, seed) -> state
    run(state) -> outputs    work(case) -> bytes, flops        tolerance(case)
"""
from __future__ import annotations

import functools
import math

import numpy as np
import torch

from paper_2608_04074_b200 import cache_format, synth, workloads
from paper_2608_04074_b200.binding import Context
from paper_2608_04074_b200.runtime import BandedCache, PagedCache

PAGE = cache_format.PAGE_TOKENS
DEV = "cuda:0"
HQ_HKV_D = {"qwen3_8b": (32, 8, 128), "gpt_oss_20b": (64, 8, 64)}
MAX_TOKEN_DIMS = 64 * 65536 * 128          # batch x length x head dimension of the largest listed decode
N_SINK, N_REC, BLOCK = 64, 256, 8          # BF16 band of the deployed format


def _step(name, model, fmt, batch, seq_len, *, append=True, ragged=False, sink=False, out="fp32"):
    return {"name": name, "kind": "step", "model": model, "format": fmt, "batch": batch, "seq_len": seq_len,
            "append": append, "ragged": ragged, "sink": sink, "out": out}


def _prefill(name, model, fmt, tokens, seqs):
    return {"name": name, "kind": "prefill", "model": model, "format": fmt, "tokens": tokens, "seqs": seqs}


def listed():
    return [
        # interactive single user, short context: nothing but latency and launches
        _step("step_b1_s777", "qwen3_8b", "plain", 1, 777),
        # small-batch serving step at medium context: the benchmark's workload
        _step("step_b8_s16384", "qwen3_8b", "plain", 8, 16384),
        # continuous batching: 128 sequences of log-normal length (1 K .. 128 K), one token each
        _step("step_mix128", "qwen3_8b", "plain", 128, 8192, ragged=True, out="bf16"),
        # long-context batch: the largest cache of the sweep (2.1 GB of indices)
        _step("decode_b64_s65536", "qwen3_8b", "plain", 64, 65536, append=False, out="bf16"),
        # full-attention layer of a model with 8 query heads per KV head, d = 64 and learned sink logits
        _step("sink_gptoss_b16_s65536", "gpt_oss_20b", "plain", 16, 65536, append=False, sink=True, out="bf16"),
        # key format with a per-token scale, odd length
        _step("scaled_b32_s8191", "qwen3_8b", "scaled", 32, 8191),
        # the paper's deployed format: scaled keys, INT2 values, BF16 sink-plus-recent band
        {"name": "deployed_band_b64_s32768", "kind": "band", "model": "qwen3_8b", "format": "deployed", "batch": 64,
         "seq_len": 32768, "out": "bf16"},
        # prompt encoding: four prompts of 8192 tokens in one call
        _prefill("prefill_32768", "qwen3_8b", "plain", 32768, 4),
        # one chunk of a chunked prefill, ragged size, deployed format
        _prefill("prefill_deployed_4099", "qwen3_8b", "deployed", 4099, 1),
        # one prompt of the d = 64 model
        _prefill("prefill_gptoss_8191", "gpt_oss_20b", "plain", 8191, 1),
        # sliding-window layer (every other layer of that model), which stays on the BF16 cache
        {"name": "window128_gptoss_b16", "kind": "window", "model": "gpt_oss_20b", "batch": 16, "seq_len": 8192,
         "window": 128, "out": "bf16"},
        # step whose inputs and outputs live in pinned host memory
        {"name": "host_gptoss_b4_s5001", "kind": "host", "model": "gpt_oss_20b", "batch": 4, "seq_len": 5001},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["step", "step", "step", "band", "prefill", "prefill", "window", "host"])
    model = "qwen3_8b" if kind == "band" else rng.choice(["qwen3_8b", "gpt_oss_20b"])
    d = HQ_HKV_D[model][2]
    fmt = rng.choice(["plain", "scaled", "deployed"]) if model == "qwen3_8b" else "plain"
    if kind == "prefill":
        tokens = _log_int(rng, 5, 32768)
        return {"kind": kind, "model": model, "format": fmt, "tokens": tokens, "seqs": min(rng.choice([1, 1, 2, 7]), tokens)}
    if kind == "window":
        return {"kind": kind, "model": "gpt_oss_20b", "batch": _log_int(rng, 1, 64), "seq_len": _log_int(rng, 100, 8192),
                "window": rng.choice([128, 128, 1024]), "out": rng.choice(["fp32", "bf16"])}
    batch = _log_int(rng, 1, 16 if kind == "host" else 128)
    seq_len = _log_int(rng, 512 if kind == "band" else 50, min(131072, MAX_TOKEN_DIMS // (batch * d) // (4 if kind == "band" else 2)))
    if kind == "host":
        return {"kind": kind, "model": model, "batch": batch, "seq_len": seq_len}
    if kind == "band":
        return {"kind": kind, "model": model, "format": "deployed", "batch": batch, "seq_len": seq_len,
                "out": rng.choice(["fp32", "bf16"])}
    return {"kind": kind, "model": model, "format": fmt, "batch": batch, "seq_len": seq_len,
            "append": rng.random() < 0.8, "ragged": rng.random() < 0.4, "sink": fmt != "deployed" and model == "gpt_oss_20b",
            "out": rng.choice(["fp32", "bf16"])}


# ------------------------------------------------------------------------------------------------ a loaded model
class _Model:
    """Calibrated layer of one model shape: what an engine loads once, whatever it is then asked to do."""

    def __init__(self, name, key_scale):
        make = workloads.qwen3_8b if name == "qwen3_8b" else workloads.gpt_oss_20b
        wl = make(batch=1, seq_len=1024, calib_tokens=2048, lloyd_iters=4)
        laws = wl.laws()
        wl.calib_queries_for_values = 256
        self.shape = s = wl.shape
        self.ctx = Context(s.n_q_heads, s.n_kv_heads, s.head_dim)
        self.ctx.novakv_load_calibration(0, wl.calibration(laws, key_scale=key_scale))
        to = lambda a: torch.from_numpy(np.ascontiguousarray(a)).to(DEV)
        self.kf, self.vf = to(laws.key_factor.astype(np.float32)), to(laws.value_factor.astype(np.float32))
        self.qf = to((laws.query_factor * np.repeat(laws.query_gain, s.hg)[:, None, None]).astype(np.float32))
        self.out_ch, self.heavy_ch = to(laws.outlier_channels), to(laws.heavy_channels)
        std = np.sqrt((laws.key_factor ** 2).sum(axis=1))                                      # [Hkv][d]
        self.heavy_std = to(np.take_along_axis(std, laws.heavy_channels, axis=1).astype(np.float32))

    def tokens(self, gen, n):
        """n new keys and values, bf16 [n][Hkv][d], of the workload's law."""
        s = self.shape
        z = lambda *size: torch.randn(size, generator=gen, device=DEV)
        k = torch.bmm(z(s.n_kv_heads, n, s.head_dim), self.kf)
        v = torch.bmm(z(s.n_kv_heads, n, s.head_dim), self.vf)
        nh = self.heavy_ch.shape[1]
        if nh:                                                                                   # Student-t, 4 degrees
            t = z(s.n_kv_heads, n, nh) / (z(4, s.n_kv_heads, n, nh).square().mean(0).sqrt())
            k.scatter_(2, self.heavy_ch[:, None, :].expand(-1, n, -1), t * self.heavy_std[:, None, :])
        if self.out_ch.shape[1]:
            idx = self.out_ch[:, None, :].expand(-1, n, -1)
            k.scatter_(2, idx, k.gather(2, idx) * 10.0)
        return tuple(x.transpose(0, 1).to(torch.bfloat16).contiguous() for x in (k, v))

    def queries(self, gen, n):
        s = self.shape
        q = torch.bmm(torch.randn((s.n_q_heads, n, s.head_dim), generator=gen, device=DEV), self.qf)
        return q.transpose(0, 1).to(torch.bfloat16).contiguous()


@functools.lru_cache(maxsize=None)
def _model(name, key_scale):
    return _Model(name, key_scale)


def _i32(a):
    return torch.from_numpy(np.ascontiguousarray(a, dtype=np.int32)).to(DEV)


def _gen(seed):
    return torch.Generator(device=DEV).manual_seed(int(seed))


def _lengths(case):
    if case.get("ragged"):
        m = case["seq_len"]
        hi = min(131072, MAX_TOKEN_DIMS // (HQ_HKV_D[case["model"]][2] * case["batch"]))
        return synth.lognormal_lengths(77, case["batch"], median=m, lo=max(1, m // 8), hi=max(m, min(16 * m, hi)))
    return np.full(case["batch"], case["seq_len"], np.int32)


def _paged(model, fmt, lens, capacity, seed):
    return PagedCache(model.ctx, lens, capacity_tokens=capacity, seed=seed % 100003, device=DEV,
                      key_scale=fmt == "scaled", int2_values=fmt == "deployed")


def _fill(model, fmt, cache, lens, gen):
    """Sequences of encoded tokens: one sequence of up to 32768 tokens is drawn and encoded, and every sequence of the
    cache gets a stretch of its pages (at pages of its own)."""
    n = min(int(lens.max()), 32768)
    n = (n + PAGE - 1) // PAGE * PAGE
    src = _paged(model, fmt, np.array([n], np.int32), None, 1)
    for t0 in range(0, n, 16384):
        m = min(16384, n - t0)
        k, v = model.tokens(gen, m)
        src.append(0, k, v, torch.zeros(m, dtype=torch.int32, device=DEV),
                   torch.arange(t0, t0 + m, dtype=torch.int32, device=DEV))
    n_pages = n // PAGE
    take, put = [], []
    for b, length in enumerate(lens):
        p = (int(length) + PAGE - 1) // PAGE
        take.append(src.page_table_host[0][(np.arange(p) + 37 * b) % n_pages])
        put.append(cache.page_table_host[b][:p])
    take, put = (torch.from_numpy(np.concatenate(x).astype(np.int64)).to(DEV) for x in (take, put))
    for name in ("k_pages", "v_pages", "k_scales", "v_meta"):
        a, b = getattr(src, name), getattr(cache, name)
        if a is not None:
            for i in range(0, len(put), 16384):
                b[put[i:i + 16384]] = a[take[i:i + 16384]]


def _sink_logits(model):
    return torch.linspace(-3.0, 3.0, model.shape.n_q_heads, device=DEV)


def _out(model, case):
    s = model.shape
    return torch.zeros((case["batch"], s.n_q_heads, s.head_dim), device=DEV,
                       dtype=torch.float32 if case.get("out", "fp32") == "fp32" else torch.bfloat16)


def prepare(case, seed):
    model = _model(case["model"], case.get("format", "plain") != "plain")
    gen = _gen(seed)
    return {"case": case, "model": model, **_PREPARE[case["kind"]](model, case, seed, gen)}


def _prepare_step(model, case, seed, gen):
    lens = _lengths(case)
    cache = _paged(model, case["format"], lens, lens + 1, seed)
    _fill(model, case["format"], cache, lens, gen)
    b = case["batch"]
    k, v = model.tokens(gen, b)
    return {"cache": cache, "q": model.queries(gen, b), "k": k, "v": v, "tok_seq": _i32(np.arange(b)), "tok_pos": _i32(lens),
            "out": _out(model, case), "sink": _sink_logits(model) if case["sink"] else None}


def _prepare_band(model, case, seed, gen):
    b, n = case["batch"], case["seq_len"]
    # a sequence in the middle of decoding: sink full, ring between N_REC and N_REC + BLOCK - 1, the rest quantised
    ring = N_REC + np.random.RandomState(seed % (1 << 31)).randint(0, BLOCK, b)
    quant = np.maximum(n - N_SINK - ring, 0).astype(np.int32)
    cache = BandedCache(model.ctx, b, n + PAGE, N_SINK, N_REC, BLOCK, seed=seed % 100003, device=DEV, int2_values=True)
    _fill(model, "deployed", cache.paged, quant + N_SINK, gen)
    rows = min(b * cache.cap, 8192)
    k, v = model.tokens(gen, rows)
    pick = (torch.arange(b * cache.cap, device=DEV) * 31) % rows
    cache.band_k.view(-1, *k.shape[1:]).copy_(k[pick])
    cache.band_v.view(-1, *v.shape[1:]).copy_(v[pick])
    cache.paged.seq_lens.copy_(_i32(quant + N_SINK))
    k, v = model.tokens(gen, b)
    meta = np.stack([np.full(b, N_SINK), (np.arange(b) * 13) % cache.ring_cap, ring], axis=1)
    return {"cache": cache, "q": model.queries(gen, b), "k": k, "v": v, "out": _out(model, case),
            "meta0": _i32(meta), "quant0": _i32(quant)}


def _prepare_prefill(model, case, seed, gen):
    n, s = case["tokens"], case["seqs"]
    lens = np.full(s, n // s, np.int32)
    lens[: n % s] += 1
    cache = _paged(model, case["format"], np.zeros(s, np.int32), lens, seed)
    k, v = model.tokens(gen, n)
    return {"cache": cache, "k": k, "v": v, "tok_seq": _i32(np.repeat(np.arange(s), lens)),
            "tok_pos": _i32(np.concatenate([np.arange(m) for m in lens]))}


def _prepare_window(model, case, seed, gen):
    s, b = model.shape, case["batch"]
    table, n_pages = synth.shuffled_page_table(seed % 100003, np.full(b, case["seq_len"], np.int32), PAGE)
    k, v = model.tokens(gen, 64 * PAGE)
    pick = (torch.arange(n_pages, device=DEV) * 29) % 64
    pool = lambda x: x.view(64, PAGE, s.n_kv_heads, s.head_dim).transpose(1, 2)[pick].contiguous()
    ws = torch.empty(model.ctx.novakv_bf16_workspace_bytes(b, table.shape[1]), dtype=torch.uint8, device=DEV)
    return {"k": pool(k), "v": pool(v), "table": _i32(table), "lens": _i32(np.full(b, case["seq_len"])), "ws": ws,
            "q": model.queries(gen, b), "out": _out(model, case)}


def _prepare_host(model, case, seed, gen):
    st = _prepare_step(model, dict(case, format="plain", sink=False), seed, gen)
    b, s = case["batch"], model.shape
    pin = {x: st.pop(x).cpu().pin_memory() for x in ("q", "k", "v", "tok_seq", "tok_pos", "out")}
    staging = torch.empty(model.ctx.novakv_step_staging_bytes(b, b), dtype=torch.uint8, device=DEV)
    return {**st, **pin, "staging": staging}


_PREPARE = {"step": _prepare_step, "band": _prepare_band, "prefill": _prepare_prefill, "window": _prepare_window,
            "host": _prepare_host}


# ------------------------------------------------------------------------------------------------ one pass
def run(state):
    return _RUN[state["case"]["kind"]](state)


def _run_step(st):
    cache = st["cache"]
    if st["case"]["append"]:
        cache.append(0, st["k"], st["v"], st["tok_seq"], st["tok_pos"])
    out = cache.decode(0, st["q"], out=st["out"], sink_logits=st["sink"])
    if not st["case"]["append"]:
        return {"out": out}
    return {"out": out, "k_pages": cache.k_pages, "v_pages": cache.v_pages, "seq_lens": cache.seq_lens}


def _run_band(st):
    # the step starts from the same band state in every pass (as after a draft token was rejected)
    cache = st["cache"]
    cache.band_meta.copy_(st["meta0"])
    cache.quant_lens.copy_(st["quant0"])
    cache.append_step(0, st["k"], st["v"], mirror=False)
    return {"out": cache.decode(0, st["q"], out=st["out"]), "meta": cache.band_meta, "quant_lens": cache.quant_lens,
            "k_pages": cache.paged.k_pages, "v_pages": cache.paged.v_pages, "k_scales": cache.paged.k_scales,
            "v_meta": cache.paged.v_meta}


def _run_prefill(st):
    cache = st["cache"]
    cache.append(0, st["k"], st["v"], st["tok_seq"], st["tok_pos"])
    out = {"k_pages": cache.k_pages, "v_pages": cache.v_pages, "seq_lens": cache.seq_lens}
    if cache.k_scales is not None:
        out["k_scales"] = cache.k_scales
    if cache.v_meta is not None:
        out["v_meta"] = cache.v_meta
    return out


def _run_window(st):
    st["model"].ctx.novakv_bf16_decode_attention(st["q"], st["k"], st["v"], st["table"], st["lens"], st["out"], st["ws"],
                                                 window=st["case"]["window"])
    return st["out"]


def _run_host(st):
    cache = st["cache"]
    st["model"].ctx.novakv_step_host(0, st["k"], st["v"], st["tok_seq"], st["tok_pos"], st["q"], cache.k_pages, cache.v_pages,
                                     cache.page_table, cache.seq_lens, st["out"], st["staging"], cache.workspace)
    return {"out": st["out"], "k_pages": cache.k_pages, "v_pages": cache.v_pages, "seq_lens": cache.seq_lens}


_RUN = {"step": _run_step, "band": _run_band, "prefill": _run_prefill, "window": _run_window, "host": _run_host}


# ------------------------------------------------------------------------------------------------ what it cannot do without
def work(case):
    hq, hkv, d = HQ_HKV_D[case["model"]]
    L = d // 4
    # per token and KV head: index bytes of both sides, and the per-token metadata of the optional formats
    meta = {"plain": 0, "scaled": 2, "deployed": 6}[case.get("format", "plain")]
    read_tables = hkv * (2 * d * d * 4 + 2 * L * 256 * 4 * 4)          # two transforms, two codebooks, binary32
    encode = lambda n: (n * hkv * (2 * d * 2 + 2 * L + meta) + read_tables,
                        n * hkv * 2 * (2 * d * d + 2 * 256 * d))       # transform, and inner products with 256 codewords per group
    if case["kind"] == "prefill":
        nbytes, flops = encode(case["tokens"])
        return {"bytes": nbytes, "flops": flops}
    b = case["batch"]
    qo = b * hq * d * (2 + (4 if case.get("out", "fp32") == "fp32" else 2))
    if case["kind"] == "window":
        n = b * min(case["seq_len"], case["window"])
        return {"bytes": n * hkv * 2 * d * 2 + qo, "flops": 4 * n * hq * d}
    n = int(_lengths(case).astype(np.int64).sum())
    nbytes, flops = n * hkv * (2 * L + meta) + read_tables + qo, 4 * n * hq * d
    if case["kind"] == "band":
        nbytes += b * (N_SINK + N_REC) * hkv * d * 2 * 2
    if case.get("append", True):
        eb, ef = encode(b)
        nbytes, flops = nbytes + eb, flops + ef
    return {"bytes": nbytes, "flops": flops}


# (rel, max) of binary32 outputs against the same attention in binary64 on the same cache, largest seen over the listed and
# drawn cases: at d = 128 the binary16 score-table entries and softmax weights, at d = 64 the softmax weights, in the
# deployed format also the rounded weights of the INT2 levels, in the sliding-window kernel binary32 sums
_SEEN = {("plain", 128): (2.7e-4, 2.7e-3), ("plain", 64): (6.3e-5, 8.0e-4), ("scaled", 128): (2.7e-4, 3.0e-3),
         ("deployed", 128): (5.4e-4, 3.3e-3), ("window", 64): (4.3e-7, 7.7e-6)}
_BF16_ROUNDING = (1.7e-3, 3.9e-3)          # of the output alone


def tolerance(case):
    """Four times what is seen against binary64.  Index bytes, scales and lengths are whole values and stay the same."""
    if case["kind"] == "prefill":
        return "exact"
    fmt = "window" if case["kind"] == "window" else case.get("format", "plain")
    rel, biggest = _SEEN[fmt, HQ_HKV_D[case["model"]][2]]
    if case.get("out") == "bf16":
        rel, biggest = max(rel, _BF16_ROUNDING[0]), max(biggest, _BF16_ROUNDING[1])
    return {"rel": 4 * rel, "max": 4 * biggest}
