"""Host-buffer step.  Without new tokens: between the kernel that gathers the queries and the one that transforms them there is
no append, and the transform must not read the staging buffer before the gather has written it.  The gather takes long enough
for a premature read to see the queries of the step before (64 sequences: half a megabyte over the bus).  Equal to the device
call bit for bit.  With new tokens: steps on both sides of the line between the append kernel and the prompt encoder, which
both let the query transform start as soon as the gather is done, and inputs of more than one pass of the gather's grid."""
import numpy as np
import pytest

from gpu_common import Case
from paper_2608_04074_b200 import workloads

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def cases():
    made = {}

    def get(model):
        if model not in made:
            make = workloads.qwen3_8b if model == "qwen" else workloads.gpt_oss_20b
            made[model] = Case(make(batch=1, seq_len=1024, calib_tokens=2048, lloyd_iters=4))
        return made[model]
    return get


@pytest.mark.parametrize("model", ["qwen", "gptoss"])
def test_step_without_new_tokens(cases, model):
    from paper_2608_04074_b200.runtime import PagedCache
    case = cases(model)
    ctx, batch, n = case.ctx, 64, 100
    cache = PagedCache(ctx, np.zeros(batch, np.int32), capacity_tokens=np.full(batch, n, np.int32), seed=3)
    k, v, q = case.draw(2100, batch * n, 8 * batch)
    dev = lambda a, dtype=torch.int32: torch.from_numpy(np.ascontiguousarray(a)).to(dtype).cuda()
    cache.append(0, dev(k, torch.bfloat16), dev(v, torch.bfloat16), dev(np.repeat(np.arange(batch), n)),
                 dev(np.tile(np.arange(n), batch)))
    qs = torch.from_numpy(q.reshape(8, batch, ctx.n_q_heads, ctx.head_dim)).to(torch.bfloat16)
    expected = [cache.decode(0, x.cuda()).cpu() for x in qs]
    pinned = [x.clone().pin_memory() for x in qs]
    out = torch.empty(expected[0].shape, dtype=torch.float32).pin_memory()
    staging = torch.empty(ctx.novakv_step_staging_bytes(batch, 0), dtype=torch.uint8, device="cuda")
    for x, ref in zip(pinned, expected):
        out.fill_(float("nan"))
        ctx.novakv_step_host(0, None, None, None, None, x, cache.k_pages, cache.v_pages, cache.page_table, cache.seq_lens,
                             out, staging, cache.workspace)
        assert torch.equal(out, ref)
    assert ctx.novakv_last_device_status() == 0


@pytest.mark.parametrize("offset", [0, 2])               # elements off the 16-byte boundary: 4-byte words across the bus
@pytest.mark.parametrize("batch", [3, "line", "line + 1", 130, 257, 601])
@pytest.mark.parametrize("model", ["qwen", "gptoss"])
def test_step_equals_append_and_decode(cases, model, batch, offset):
    from paper_2608_04074_b200.runtime import PagedCache
    case = cases(model)
    ctx, line = case.ctx, case.ctx.novakv_debug_append_kernel_tokens()
    batch = {"line": line, "line + 1": line + 1}.get(batch, batch)
    lens = (37 * np.arange(batch) % 200).astype(np.int32)
    k, v, q = case.draw(2200 + batch, batch, batch)
    seq = np.random.RandomState(3).permutation(batch).astype(np.int32)
    new = [torch.from_numpy(x).to(torch.bfloat16) for x in (k, v, q)] + [torch.from_numpy(x) for x in (seq, lens[seq])]
    if batch == 601:                                     # one pass: 256 threads in 8 blocks an SM, 16 bytes each
        sms = torch.cuda.get_device_properties(0).multi_processor_count
        assert model == "gptoss" or sum(x.numel() * x.element_size() for x in new) > 8 * sms * 256 * 16

    def cache():
        c = PagedCache(ctx, lens, capacity_tokens=lens + 1, seed=5)
        gen = torch.Generator(device="cuda").manual_seed(6)
        for pool in (c.k_pages, c.v_pages):
            pool.copy_(torch.randint(0, 256, pool.shape, generator=gen, dtype=torch.uint8, device="cuda"))
        return c

    a, b = cache(), cache()
    kd, vd, qd, sd, pd = (x.cuda() for x in new)
    a.append(0, kd, vd, sd, pd)
    torch.cuda.synchronize()
    expected = a.decode(0, qd).cpu()
    pinned = []
    for x in new:
        p = torch.empty(x.numel() + offset, dtype=x.dtype).pin_memory()[offset:].view(x.shape)
        pinned.append(p.copy_(x))
        assert p.data_ptr() % 16 == offset * x.element_size() % 16
    out = torch.full(expected.shape, float("nan")).pin_memory()
    staging = torch.empty(ctx.novakv_step_staging_bytes(batch, batch), dtype=torch.uint8, device="cuda")
    ctx.novakv_step_host(0, pinned[0], pinned[1], pinned[3], pinned[4], pinned[2], b.k_pages, b.v_pages, b.page_table,
                         b.seq_lens, out, staging, b.workspace)
    assert torch.equal(out, expected)
    for x, y in ((a.k_pages, b.k_pages), (a.v_pages, b.v_pages), (a.seq_lens, b.seq_lens)):
        assert torch.equal(x, y)
    assert ctx.novakv_last_device_status() == 0
