"""Batches on both sides of the sizes at which a call takes another way: the scan's own prefixes (up to 511 sequences; warps of
32), and the append kernel or the prompt encoder (two passes of eight tokens for every chunk that fits on the machine, which
depends on the KV heads).  Outputs: 2e-3 of the largest
(check_output); indices and scales equal the oracle's (check_indices)."""
import numpy as np
import pytest

from gpu_common import Case, check_indices, check_output
from paper_2608_04074_b200 import cache_format, synth, workloads

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

NOVAKV_DEV_BAD_LENGTH = 2


@pytest.fixture(scope="module")
def cases():
    made = {}

    def get(name, scaled=False):
        if (name, scaled) not in made:
            make = workloads.qwen3_8b if name == "qwen" else workloads.gpt_oss_20b
            made[name, scaled] = Case(make(batch=1, seq_len=1024, calib_tokens=2048, lloyd_iters=4), key_scale=scaled)
        return made[name, scaled]
    return get


@pytest.mark.parametrize("batch", [1, 31, 32, 33, 510, 511, 512])
@pytest.mark.parametrize("name", ["qwen", "gptoss"])
def test_prefixes(cases, name, batch):
    from paper_2608_04074_b200.runtime import PagedCache
    case = cases(name)
    lens = (29 * np.arange(batch) % 150 + 1).astype(np.int32)
    lens[1::7] = 0                                                     # empty ones in every warp
    if batch > 1:
        lens[-1] = 0
    cache = PagedCache(case.ctx, lens, seed=4)
    k, v, _ = case.draw(700, 400, 1)
    e = case.oracle.encode(k.astype(np.float64), v.astype(np.float64), with_gaps=False)
    part = [(e["kidx"][b % 200:b % 200 + n], e["vidx"][b % 200:b % 200 + n]) for b, n in enumerate(lens)]
    cache.store_logical_batch([(b, 0, *p) for b, p in enumerate(part) if lens[b]])
    _, _, q = case.draw(701, 1, batch)
    qd = torch.from_numpy(q).to(torch.bfloat16).cuda()
    out = cache.decode(0, qd).cpu().numpy()
    assert case.ctx.novakv_last_device_status() == 0
    for b in sorted({0, 1, batch // 2, batch - 2, batch - 1, *range(29, min(batch, 36)), *range(0, batch, 61)}):
        if 0 <= b < batch:
            if lens[b]:
                check_output(out[b], case.oracle.decode(q[b].astype(np.float64), *part[b]))
            else:
                assert not out[b].any()
    # a length beyond the row's capacity is clamped and reported
    cache.seq_lens[int(np.argmax(lens))] = cache.page_table.shape[1] * 64 + 1
    cache.decode(0, qd)
    assert case.ctx.novakv_last_device_status() == NOVAKV_DEV_BAD_LENGTH


def _append_or_prompt(case, fmt, n):
    from paper_2608_04074_b200.runtime import PagedCache
    cache = PagedCache(case.ctx, np.zeros(2, np.int32), capacity_tokens=np.array([n, n]), seed=6, key_scale=fmt == "scaled",
                       int2_values=fmt == "deployed")
    k, v, _ = case.draw(900 + n, n, 1)
    dev = lambda a: torch.from_numpy(a).to(torch.bfloat16).cuda()
    seq = (np.arange(n) % 2).astype(np.int32)
    cache.append(0, dev(k), dev(v), torch.from_numpy(seq).cuda(), torch.from_numpy((np.arange(n) // 2).astype(np.int32)).cuda())
    assert case.ctx.novakv_last_device_status() == 0
    assert cache.seq_lens.tolist() == [(n + 1) // 2, n // 2]
    k64, v64 = k.astype(np.float64), v.astype(np.float64)
    e = (case.oracle.encode if fmt == "plain" else case.oracle.encode_scaled)(k64, v64)
    for s in (0, 1):
        kidx, vidx = cache.load_logical(s, 0, int((seq == s).sum()))
        mine = {x: y[seq == s] for x, y in e.items()}
        check_indices(kidx, mine, "k")
        if fmt == "deployed":
            codes, meta = case.oracle.encode_values_int2(v64)
            assert np.array_equal(vidx, cache_format.pack_int2(codes)[seq == s])
            assert np.array_equal(cache.load_value_meta(s, 0, len(vidx)), meta[seq == s].astype(np.float32))
        else:
            check_indices(vidx, mine, "v")
        if fmt != "plain":
            assert np.array_equal(cache.load_scales(s, 0, len(kidx)), mine["kscale"].astype(np.float32))


@pytest.mark.parametrize("n", [64, 65, 192, 193, "line", "line + 1"])
@pytest.mark.parametrize("name,fmt", [("qwen", "plain"), ("qwen", "scaled"), ("qwen", "deployed"), ("gptoss", "plain"), ("gptoss", "scaled")])
def test_append_or_prompt(cases, name, fmt, n):
    case = cases(name, fmt != "plain")
    line = case.ctx.novakv_debug_append_kernel_tokens()
    _append_or_prompt(case, fmt, {"line": line, "line + 1": line + 1}.get(n, n))


@pytest.mark.parametrize("fmt", ["plain", "deployed"])
@pytest.mark.parametrize("hkv,d", [(1, 64), (1, 128), (2, 128), (3, 128), (4, 128), (16, 64), (16, 128)])
def test_append_or_prompt_by_heads(hkv, d, fmt):
    wl = workloads.Workload("heads", synth.LayerShape(hkv, hkv, d), np.array([1024], np.int32), 7, n_outlier=2, calib_tokens=1024,
                            calib_queries_for_values=128, lloyd_iters=2)
    case = Case(wl, key_scale=fmt != "plain")
    line = case.ctx.novakv_debug_append_kernel_tokens()
    chunks = max(1, 5 * torch.cuda.get_device_properties(0).multi_processor_count // (d // 16 * hkv * 2))
    assert line == max(64 if d == 128 else 192, min(256, 16 * chunks))
    for n in (line // 2 + 3, line, line + 1):
        _append_or_prompt(case, fmt, n)
    case.ctx.close()


@pytest.mark.parametrize("sink", [False, True])
@pytest.mark.parametrize("beyond", [0, 1])
def test_merge_in_halves(cases, beyond, sink):
    """More sequences than four for every SM's block of the merge kernel: two blocks an SM, each with half of the run."""
    from paper_2608_04074_b200.runtime import PagedCache
    case = cases("qwen")
    batch = 4 * (torch.cuda.get_device_properties(0).multi_processor_count // case.ctx.n_kv_heads) + beyond
    lens = (31 * np.arange(batch) % 170).astype(np.int32)              # the first is empty
    lens[-1] = 0
    lens[2] = 2000                                                     # one with many pieces
    cache = PagedCache(case.ctx, lens, seed=8)
    k, v, _ = case.draw(710, 2000, 1)
    e = case.oracle.encode(k.astype(np.float64), v.astype(np.float64), with_gaps=False)
    part = [(e["kidx"][f:f + n], e["vidx"][f:f + n]) for f, n in ((13 * b % 1800 if n <= 170 else 0, n) for b, n in enumerate(lens))]
    cache.store_logical_batch([(b, 0, *p) for b, p in enumerate(part) if lens[b]])
    _, _, q = case.draw(711, 1, batch)
    logits = np.linspace(-3.0, 3.0, case.ctx.n_q_heads).astype(np.float32)
    out = cache.decode(0, torch.from_numpy(q).to(torch.bfloat16).cuda(),
                       sink_logits=torch.from_numpy(logits).cuda() if sink else None).cpu().numpy()
    assert case.ctx.novakv_last_device_status() == 0
    for b, n in enumerate(lens):
        if n == 0:
            assert not out[b].any()
            continue
        args = (q[b].astype(np.float64), *part[b])
        check_output(out[b], case.oracle.decode_sink(*args, logits.astype(np.float64)) if sink else case.oracle.decode(*args))
