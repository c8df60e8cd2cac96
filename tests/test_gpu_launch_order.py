"""Calls in a row on one stream, nothing between them: the query transform runs beside the kernel in front, and must leave
everything alone that this kernel may still read.  Each pair of calls shares memory the way scratch may be shared; the same
calls with buffers of their own and a wait between them give the expected bits."""
import numpy as np
import pytest

from gpu_common import Case
from paper_2608_04074_b200 import synth, workloads

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

TIMES = 20


def _dev(a, dtype=torch.int32):
    return torch.from_numpy(np.ascontiguousarray(a)).to(dtype).cuda()


def _scratch(n):
    return torch.zeros(int(n), dtype=torch.uint8, device="cuda")


@pytest.fixture(scope="module")
def cases():
    made = {}

    def get(name, scaled=False):
        if (name, scaled) not in made:
            make = workloads.qwen3_8b if name == "qwen" else workloads.gpt_oss_20b
            made[name, scaled] = Case(make(batch=1, seq_len=1024, calib_tokens=2048, lloyd_iters=4), key_scale=scaled)
        return made[name, scaled]
    return get


def _cache(case, lens, seed, **kw):
    """A cache of random indices (any byte is a valid index) with its queries."""
    from paper_2608_04074_b200.runtime import PagedCache
    cache = PagedCache(case.ctx, lens, seed=seed, **kw)
    gen = torch.Generator(device="cuda").manual_seed(seed)
    for pool in (cache.k_pages, cache.v_pages):
        pool.copy_(torch.randint(0, 256, pool.shape, generator=gen, dtype=torch.uint8, device="cuda"))
    if cache.v_meta is not None:
        cache.v_meta.copy_(torch.rand(cache.v_meta.shape, generator=gen, device="cuda"))
    shape = (len(lens), case.ctx.n_q_heads, case.ctx.head_dim)
    return cache, torch.randn(shape, generator=gen, device="cuda").to(torch.bfloat16)


@pytest.mark.parametrize("name", ["qwen", "gptoss"])
@pytest.mark.parametrize("first", ["window", "decode"])
def test_scratch_of_the_call_in_front(cases, name, first):
    """A call whose last kernel merges partials out of its scratch, then the decode of a larger batch on the same scratch:
    the queries of the second lie where the partials of the first are."""
    case = cases(name)
    ctx, dim = case.ctx, case.ctx.n_q_heads * case.ctx.head_dim
    big, q_big = _cache(case, np.full(96, 200, np.int32), 11)
    lens = np.array([6000, 3000, 40, 0], np.int32)
    small, q_small = _cache(case, lens, 12)
    table, n_pages = synth.shuffled_page_table(13, np.maximum(lens, 1), 64)
    gen = torch.Generator(device="cuda").manual_seed(14)
    pools = [torch.randn((n_pages, ctx.n_kv_heads, 64, ctx.head_dim), generator=gen, device="cuda").to(torch.bfloat16) for _ in range(2)]
    table, lens_d = _dev(np.where(table < 0, 0, table)), _dev(lens)
    out_a, out_b = torch.empty((len(lens), ctx.n_q_heads, ctx.head_dim), device="cuda"), torch.empty((96, ctx.n_q_heads, ctx.head_dim), device="cuda")

    def calls(ws_a, ws_b, wait):
        if first == "window":
            ctx.novakv_bf16_decode_attention(q_small, *pools, table, lens_d, out_a, ws_a, window=0)
        else:
            ctx.novakv_decode_attention(0, q_small, small.k_pages, small.v_pages, small.page_table, small.seq_lens, out_a, ws_a)
        if wait:
            torch.cuda.synchronize()
        ctx.novakv_decode_attention(0, q_big, big.k_pages, big.v_pages, big.page_table, big.seq_lens, out_b, ws_b)
        return out_a.clone(), out_b.clone()

    need_a = max(ctx.novakv_bf16_workspace_bytes(len(lens), table.shape[1]), ctx.novakv_decode_workspace_bytes(len(lens)))
    need_b = ctx.novakv_decode_workspace_bytes(96)
    expected = calls(_scratch(need_a), _scratch(need_b), True)
    assert need_b > 96 * dim * 4 and expected[0].any() and expected[1].any()
    ws = _scratch(max(need_a, need_b))
    for _ in range(TIMES):
        assert all(torch.equal(x, y) for x, y in zip(calls(ws, ws, False), expected))
    assert ctx.novakv_last_device_status() == 0


@pytest.mark.parametrize("n", [33, 64, 300, 2000])
@pytest.mark.parametrize("name,fmt", [("qwen", "plain"), ("gptoss", "plain"), ("qwen", "deployed")])
def test_new_rows_in_the_scratch_of_the_decode(cases, name, fmt, n):
    """New rows whose memory becomes the scratch of the decode behind the append (a freed tensor): the append kernel and the
    prompt encoder let the query transform start before they have read them."""
    from paper_2608_04074_b200.runtime import PagedCache
    case = cases(name, fmt != "plain")
    ctx = case.ctx
    big, q = _cache(case, np.full(96, 200, np.int32), 21, int2_values=fmt == "deployed")
    cache = PagedCache(ctx, np.array([0], np.int32), capacity_tokens=np.array([n], np.int32), int2_values=fmt == "deployed")
    k, v, _ = case.draw(3100 + n, n, 1)
    rows, seq, pos = _dev(np.stack([k, v]), torch.bfloat16), _dev(np.zeros(n)), _dev(np.arange(n))
    scratch = _scratch(max(big.workspace.numel(), rows.numel() * 2))
    inside = scratch[:rows.numel() * 2].view(torch.bfloat16).view(rows.shape)
    out = torch.empty(q.shape, device="cuda")

    def calls(new, ws, wait):
        cache.k_pages.zero_(), cache.v_pages.zero_(), cache.seq_lens.zero_()
        cache.append(0, new[0], new[1], seq, pos)
        if wait:
            torch.cuda.synchronize()
        big.workspace = ws
        big.decode(0, q, out=out)
        return [x.clone() for x in (cache.k_pages, cache.v_pages, cache.seq_lens, out, cache.k_scales, cache.v_meta) if x is not None]

    expected = calls(rows, _scratch(big.workspace.numel()), True)
    assert expected[0].any()
    for _ in range(TIMES):
        inside.copy_(rows)
        assert all(torch.equal(x, y) for x, y in zip(calls(inside, scratch, False), expected))
    assert ctx.novakv_last_device_status() == 0


@pytest.mark.parametrize("fmt", ["scaled", "deployed"])
def test_band_rows_from_the_call_in_front(cases, fmt):
    """Band rows that the kernel directly before the decode call writes, having let its dependents start (here: the output of
    another decode): the band kernel has to see them."""
    from paper_2608_04074_b200.runtime import BandedCache
    case = cases("qwen", True)
    ctx = case.ctx
    other, q_other = _cache(case, np.full(32, 3000, np.int32), 31, key_scale=True)
    banded = BandedCache(ctx, 4, 2000, seed=5, key_scale=fmt == "scaled", int2_values=fmt == "deployed")
    for b, n in enumerate((1500, 700, 330, 60)):
        k, v, _ = case.draw(3200 + b, n, 1)
        banded.prefill(0, b, _dev(k, torch.bfloat16), _dev(v, torch.bfloat16))
    _, _, q = case.draw(3300, 1, 4)
    q = _dev(q, torch.bfloat16)
    rows = banded.band_v.view(-1)[:q_other.numel()].view(q_other.shape)      # the first rows of the band
    before = rows.clone()

    def calls(wait):
        rows.copy_(before)
        other.decode(0, q_other, out=rows)
        if wait:
            torch.cuda.synchronize()
        return banded.decode(0, q)

    expected = calls(True)
    rows.copy_(before)
    assert not torch.equal(banded.decode(0, q), expected)
    for _ in range(TIMES):
        assert torch.equal(calls(False), expected)
    assert ctx.novakv_last_device_status() == 0


@pytest.mark.parametrize("batch", [2, 9, 64])
def test_band_staging_in_the_scratch_of_the_decode(cases, batch):
    """The rows that leave the band are encoded out of a staging buffer; the decode that follows may use the same scratch."""
    from paper_2608_04074_b200.runtime import BandedCache
    case = cases("qwen", True)
    ctx, n_sink, n_rec, block = case.ctx, 64, 64, 8
    banded = BandedCache(ctx, batch, 1024, n_sink, n_rec, block, seed=6, int2_values=True)
    gen = torch.Generator(device="cuda").manual_seed(41)
    for band in (banded.band_k, banded.band_v):
        band.copy_(torch.randn(band.shape, generator=gen, device="cuda"))
    k, v = torch.randn((2, batch, ctx.n_kv_heads, ctx.head_dim), generator=gen, device="cuda").to(torch.bfloat16)
    q = torch.randn((batch, ctx.n_q_heads, ctx.head_dim), generator=gen, device="cuda").to(torch.bfloat16)
    p, bands = banded.paged, (banded.band_k.clone(), banded.band_v.clone())
    need = ctx.novakv_band_append_staging_bytes(batch, block), p.workspace.numel()

    def calls(staging, ws, wait):
        banded.band_k.copy_(bands[0]), banded.band_v.copy_(bands[1])
        p.k_pages.zero_(), p.v_pages.zero_(), p.seq_lens.zero_(), banded.quant_lens.zero_()
        banded.band_meta.copy_(_dev(np.tile([n_sink, 3, n_rec + block - 1], (batch, 1))))      # every sequence gives up a block
        banded._staging, p.workspace = staging, ws
        banded.append_step(0, k, v, mirror=False)
        if wait:
            torch.cuda.synchronize()
        return [x.clone() for x in (banded.decode(0, q), p.k_pages, p.v_pages, p.k_scales, p.v_meta, banded.quant_lens)]

    expected = calls(*map(_scratch, need), True)
    assert expected[1].any() and expected[-1].tolist() == [block] * batch
    shared = _scratch(max(need))
    for _ in range(TIMES):
        assert all(torch.equal(x, y) for x, y in zip(calls(shared, shared, False), expected))
    assert ctx.novakv_last_device_status() == 0
