"""Prompt encoder (more tokens per call than the append kernel takes, which the context tells) at the edges of its tiling:
256-token units of two 128-token halves, runs of units cut across (KV head, side, part of the groups) boundaries, and the
exact re-search of close decisions.  Indices, scales and (scale, zero) pairs must equal the oracle's; only float64 near-ties may
differ (gpu_common).  Where the append kernel is the witness - its bounds are derived, the encoder's measured -, the same tokens
are stored in one call and in steps of the largest size that the append kernel takes."""
import dataclasses

import numpy as np
import pytest

from gpu_common import Case, check_indices
from paper_2608_04074_b200 import synth, workloads

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


def _dev(a, dtype=None):
    t = torch.from_numpy(np.ascontiguousarray(a))
    return (t if dtype is None else t.to(dtype)).cuda()


def _make(name, key_scale):
    wl = (workloads.qwen3_8b(batch=1, seq_len=1024, calib_tokens=2048, lloyd_iters=4) if name == "qwen"
          else workloads.gpt_oss_20b(batch=1, seq_len=1024, calib_tokens=2048, lloyd_iters=4))
    return Case(dataclasses.replace(wl, calib_queries_for_values=256), key_scale=key_scale)


@pytest.fixture(scope="module")
def cases():
    return {(n, s): _make(n, s) for n in ("qwen", "gptoss") for s in (False, True)}


def _append_step(case):
    """Tokens per call of the append kernel, at most: one more and the encoder would be compared with itself."""
    step = case.ctx.novakv_debug_append_kernel_tokens()
    assert 8 <= step < 257                              # (every test of the encoder has more tokens in a call)
    return step


def _run(case, fmt, n, start, permute, holes, scale=1.0, offset=0):
    from paper_2608_04074_b200.runtime import PagedCache
    k, v, _ = case.draw(4000 + n, n, 1)
    k, v = (synth.to_bf16_representable(x * scale) for x in (k, v))
    cache = PagedCache(case.ctx, np.array([0, 0], np.int32), capacity_tokens=np.array([start + n, 64], np.int32), seed=7,
                       key_scale=fmt == "scaled", int2_values=fmt == "deployed")
    pos = start + np.arange(n, dtype=np.int32)
    seq = np.zeros(n, np.int32)
    used = np.ones(n, bool)
    if holes:
        used[::7] = False
        seq[~used] = -1
    order = synth.rng(3).permutation(n) if permute else np.arange(n)
    kd, vd = (_dev(x[order], torch.bfloat16) for x in (k, v))
    if offset:                                   # rows that start `offset` elements off a 16-byte boundary
        kd, vd = (torch.cat([x.new_zeros(offset), x.flatten()])[offset:].view(x.shape) for x in (kd, vd))
        assert kd.data_ptr() % 16 == 2 * offset
    cache.append(0, kd, vd, _dev(seq[order]), _dev(pos[order]))
    assert case.ctx.novakv_last_device_status() == 0
    assert int(cache.seq_lens[0]) == start + int(np.flatnonzero(used)[-1]) + 1 and int(cache.seq_lens[1]) == 0
    gk, gv = cache.load_logical(0, start, n)
    assert not gk[~used].any() and not gv[~used].any()
    k64, v64 = k[used].astype(np.float64), v[used].astype(np.float64)
    if fmt == "plain":
        e = case.oracle.encode(k64, v64)
    else:
        e = case.oracle.encode_scaled(k64, v64)
        assert np.array_equal(cache.load_scales(0, start, n)[used], e["kscale"])
    check_indices(gk[used], e, "k")
    if fmt == "deployed":
        from paper_2608_04074_b200 import cache_format
        codes, meta = case.oracle.encode_values_int2(v64)
        assert np.array_equal(gv[used], cache_format.pack_int2(codes))
        assert np.array_equal(cache.load_value_meta(0, start, n)[used], meta)
    else:
        check_indices(gv[used], e, "v")


@pytest.mark.parametrize("n,start,permute,holes", [
    (257, 0, False, False),      # one unit and one token of a second; whole 16-token value blocks
    (384, 64, False, False),     # the last half tile of a unit is empty
    (511, 5, False, False),      # positions off the 16-token blocks
    (512, 0, True, False),       # tokens of a warp scattered over pages
    (513, 16, False, True),      # unused entries
    (2049, 48, False, False),    # runs of units that cross head, side and group boundaries
])
@pytest.mark.parametrize("name,fmt", [("qwen", "plain"), ("gptoss", "plain"), ("qwen", "scaled"), ("gptoss", "scaled"),
                                      ("qwen", "deployed"), ("gptoss", "deployed")])
def test_prefill_edges(cases, name, fmt, n, start, permute, holes):
    _run(cases[name, fmt != "plain"], fmt, n, start, permute, holes)


@pytest.mark.parametrize("name,scale", [("qwen", 0.0), ("qwen", 1e-3), ("qwen", 64.0), ("gptoss", 1e-3), ("gptoss", 64.0)])
def test_prefill_far_from_the_codebook(cases, name, scale):
    """Inputs a thousand times smaller and 64 times larger than the calibration's (and all zero): the binary16 ranking
    is then dominated by rounding, or out of its range, and every decision rests on the exact re-search."""
    _run(cases[name, False], "plain", 300, 0, False, False, scale)


@pytest.mark.parametrize("name", ["qwen", "gptoss"])
def test_prefill_rows_without_tensor_map_alignment(cases, name):
    """New rows on a 4-byte boundary cannot be copied by a tensor map: the plain copies must give the same indices."""
    _run(cases[name, False], "plain", 600, 0, False, False, offset=2)


@pytest.mark.parametrize("n", [1, 8, 130, 256])
@pytest.mark.parametrize("name,fmt", [("qwen", "plain"), ("gptoss", "scaled"), ("qwen", "deployed")])
def test_append_rows_on_a_word_boundary(cases, name, fmt, n):
    """Batches of the append kernel's size whose rows it cannot read (16-byte loads): the same indices, at any number."""
    _run(cases[name, fmt != "plain"], fmt, n, 40, False, False, offset=2)


@pytest.mark.parametrize("n", [8, 600])
def test_append_rows_off_a_word_boundary_are_refused(cases, n):
    from paper_2608_04074_b200.binding import NovaKVError
    with pytest.raises(NovaKVError, match="invalid argument"):
        _run(cases["qwen", False], "plain", n, 0, False, False, offset=1)


@pytest.mark.parametrize("kind", ["positive", "cancelling", "wide"])
@pytest.mark.parametrize("name,fmt", [("qwen", "plain"), ("gptoss", "plain"), ("qwen", "scaled"), ("gptoss", "scaled")])
def test_prefill_bounds_hold_on_hard_inputs(cases, name, fmt, kind):
    """The bounds of the tensor core's errors are measured, not derived: inputs that strain them - all positive (every
    truncation in one direction), pairs of opposite sign (small coefficients of large rows), elements over three decades -
    must leave no index that the append kernel, whose bound is derived, decides differently."""
    from paper_2608_04074_b200.runtime import PagedCache
    case, n = cases[name, fmt != "plain"], 16384
    gen = torch.Generator(device="cuda").manual_seed(12)
    shape = (n, case.ctx.n_kv_heads, case.ctx.head_dim)
    x = torch.randn((2, *shape), generator=gen, device="cuda")
    if kind == "positive":
        x = x.abs()
    elif kind == "cancelling":
        x = torch.stack([x[..., ::2] * 4, -x[..., ::2] * 4 + x[..., 1::2] * 0.25], dim=-1).flatten(-2)
    else:
        x = x * 10.0 ** (torch.rand(x.shape, generator=gen, device="cuda") * 3 - 2)
    k, v = x.to(torch.bfloat16)
    seq, pos = torch.zeros(n, dtype=torch.int32, device="cuda"), torch.arange(n, dtype=torch.int32, device="cuda")
    stored = []
    for step in (n, _append_step(case)):
        cache = PagedCache(case.ctx, np.array([0], np.int32), capacity_tokens=np.array([n], np.int32), seed=7, key_scale=fmt == "scaled")
        for i in range(0, n, step):
            cache.append(0, k[i:i + step], v[i:i + step], seq[i:i + step], pos[i:i + step])
        assert case.ctx.novakv_last_device_status() == 0
        stored.append([y for y in (cache.k_pages, cache.v_pages, cache.k_scales) if y is not None])
    for prompt, small in zip(*stored):
        assert torch.equal(prompt, small), int((prompt != small).sum())


@pytest.mark.parametrize("first,n", [(0, 600), (299, 300), (640, 700), (1279, 2048), (2047, 2048), (3000, 3000)])
@pytest.mark.parametrize("name,fmt", [("qwen", "plain"), ("gptoss", "scaled"), ("qwen", "deployed")])
def test_prefill_leading_entries_unused(cases, name, fmt, first, n):
    """Lists that begin with `first` unused entries (first = n: nothing else): the CTAs that meet none leave, the
    others store what they always store."""
    from paper_2608_04074_b200.runtime import PagedCache
    case = cases[name, fmt != "plain"]
    k, v, _ = case.draw(4500, n, 1)
    kd, vd, pos = _dev(k, torch.bfloat16), _dev(v, torch.bfloat16), np.arange(n, dtype=np.int32)
    stored = []
    for seq in (np.where(pos < first, -1, 0), np.zeros(n)):
        cache = PagedCache(case.ctx, np.array([0], np.int32), capacity_tokens=np.array([n], np.int32), seed=7,
                           key_scale=fmt == "scaled", int2_values=fmt == "deployed")
        cache.append(0, kd, vd, _dev(seq.astype(np.int32)), _dev(pos))
        assert case.ctx.novakv_last_device_status() == 0
        stored.append([*cache.load_logical(0, 0, n), *([cache.load_scales(0, 0, n)] if fmt != "plain" else []), cache.seq_lens.cpu()])
    part, full = stored
    assert int(part[-1][0]) == (n if first < n else 0)
    for i, (p, f) in enumerate(zip(part[:-1], full[:-1])):
        assert np.array_equal(p[first:], f[first:]) and (p[:first] == (1 if i == 2 else 0)).all()


@pytest.mark.parametrize("factor", [1e-17, 1e-22, 1e-30])
@pytest.mark.parametrize("name,fmt", [("qwen", "scaled"), ("gptoss", "scaled"), ("qwen", "deployed")])
def test_prefill_squares_that_underflow(cases, name, fmt, factor):
    """Per-token scales make the format indifferent to the size of the inputs, so the error bound of the coefficients must not
    vanish with the squares of the row: the same bytes as the append kernel's, which searches binary64 coefficients."""
    from paper_2608_04074_b200.runtime import PagedCache
    case, n = cases[name, True], 16384
    gen = torch.Generator(device="cuda").manual_seed(11)
    k, v = ((torch.randn((n, case.ctx.n_kv_heads, case.ctx.head_dim), generator=gen, device="cuda") * factor).to(torch.bfloat16)
            for _ in range(2))
    k[:, :, ::16] *= 40.0                                  # a few large elements: small coefficients with large errors beside them
    seq, pos = torch.zeros(n, dtype=torch.int32, device="cuda"), torch.arange(n, dtype=torch.int32, device="cuda")
    stored = []
    for step in (n, _append_step(case)):
        cache = PagedCache(case.ctx, np.array([0], np.int32), capacity_tokens=np.array([n], np.int32), seed=7,
                           key_scale=fmt == "scaled", int2_values=fmt == "deployed")
        for i in range(0, n, step):
            cache.append(0, k[i:i + step], v[i:i + step], seq[i:i + step], pos[i:i + step])
        assert case.ctx.novakv_last_device_status() == 0
        stored.append([x for x in (cache.k_pages, cache.v_pages, cache.k_scales, cache.v_meta) if x is not None])
    for prompt, small in zip(*stored):
        assert torch.equal(prompt, small), int((prompt != small).sum())


@pytest.mark.parametrize("name,fmt", [("qwen", "plain"), ("gptoss", "scaled"), ("qwen", "deployed")])
@pytest.mark.parametrize("shift", [1, 2])
def test_prefill_pools_off_a_word_boundary(cases, name, fmt, shift):
    """The append entries take pools on any address (decode wants 16 bytes): same bytes, written one by one."""
    from paper_2608_04074_b200.runtime import PagedCache
    case, n = cases[name, fmt != "plain"], 333
    k, v, _ = case.draw(4400, n, 1)
    args = (_dev(k, torch.bfloat16), _dev(v, torch.bfloat16), _dev(np.zeros(n, np.int32)), _dev(np.arange(n, dtype=np.int32)))
    stored = []
    for off in (0, shift):
        cache = PagedCache(case.ctx, np.array([0], np.int32), capacity_tokens=np.array([n], np.int32), seed=7,
                           key_scale=fmt == "scaled", int2_values=fmt == "deployed")
        shifted = lambda x: torch.zeros(x.numel() + off, dtype=torch.uint8, device="cuda")[off:].view(x.shape)
        cache.k_pages, cache.v_pages = shifted(cache.k_pages), shifted(cache.v_pages)
        assert cache.k_pages.data_ptr() % 4 == off
        cache.append(0, *args)
        assert case.ctx.novakv_last_device_status() == 0
        stored.append((cache.k_pages.clone(), cache.v_pages.clone()))
    assert all(torch.equal(a, b) for a, b in zip(*stored))


@pytest.mark.parametrize("n", [24, 41, 57, "most"])
@pytest.mark.parametrize("name,fmt", [("qwen", "plain"), ("gptoss", "plain"), ("qwen", "scaled"), ("gptoss", "deployed")])
def test_append_batches_of_several_chunks(cases, name, fmt, n):
    """Batches that still take the append kernel but span several of its passes and chunks of the token list."""
    most = _append_step(cases[name, fmt != "plain"])
    assert most >= 57
    _run(cases[name, fmt != "plain"], fmt, most if n == "most" else n, 40, True, n == 57)


@pytest.mark.parametrize("bad", [float("nan"), float("inf"), -float("inf")])
@pytest.mark.parametrize("name,fmt", [("qwen", "plain"), ("gptoss", "plain"), ("qwen", "scaled"), ("gptoss", "deployed")])
def test_prefill_token_that_is_not_finite(cases, name, fmt, bad):
    """One element of one token is not a number: its distances are not either, and a scan that keeps a smaller distance
    keeps index 0 - what the append kernel stores.  (INT2 values: the same bytes as the append kernel's.)  The other tokens
    do not notice."""
    from paper_2608_04074_b200.runtime import PagedCache
    case, n, t = cases[name, fmt != "plain"], 300, 130
    k, v, _ = case.draw(4300, n, 1)

    def stored(bad_value, step):
        kb, vb = k.copy(), v.copy()
        if bad_value is not None:
            kb[t, :, 5] = vb[t, :, 5] = bad_value
        cache = PagedCache(case.ctx, np.array([0], np.int32), capacity_tokens=np.array([n], np.int32), seed=7,
                           key_scale=fmt == "scaled", int2_values=fmt == "deployed")
        for i in range(0, n, step):
            j = min(i + step, n)
            cache.append(0, _dev(kb[i:j], torch.bfloat16), _dev(vb[i:j], torch.bfloat16), _dev(np.zeros(j - i, np.int32)),
                         _dev(np.arange(i, j, dtype=np.int32)))
        assert case.ctx.novakv_last_device_status() == 0
        return [*cache.load_logical(0, 0, n), *([cache.load_scales(0, 0, n)] if fmt != "plain" else [])]

    clean, prompt, small = stored(None, n), stored(bad, n), stored(bad, min(150, _append_step(case)))
    for c, p, s in zip(clean, prompt, small):
        assert np.array_equal(p[t], s[t])
        assert np.array_equal(np.delete(p, t, 0), np.delete(c, t, 0))
    if np.isnan(bad):
        assert not prompt[0][t].any() and (fmt == "deployed" or not prompt[1][t].any())
