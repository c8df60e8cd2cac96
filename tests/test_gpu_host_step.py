"""Host-buffer step without new tokens: between the kernel that gathers the queries and the one that transforms them there is
no append, and the transform must not read the staging buffer before the gather has written it.  The gather takes long enough
for a premature read to see the queries of the step before (64 sequences: half a megabyte over the bus).  Equal to the device
call bit for bit."""
import numpy as np
import pytest

from gpu_common import Case
from paper_2608_04074_b200 import workloads

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.mark.parametrize("model", ["qwen", "gptoss"])
def test_step_without_new_tokens(model):
    from paper_2608_04074_b200.runtime import PagedCache
    make = workloads.qwen3_8b if model == "qwen" else workloads.gpt_oss_20b
    case = Case(make(batch=1, seq_len=1024, calib_tokens=2048, lloyd_iters=4))
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
