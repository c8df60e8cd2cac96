"""Prompt encoder with waits that give up early: the call returns, says so in the status word, leaves alone every byte that
does not belong to its tokens, and the next call with the usual limit stores what it always stores.  Which waits run out
depends on the limit and on timing; whichever they are, the same has to hold."""
import numpy as np
import pytest

from gpu_common import Case
from paper_2608_04074_b200 import workloads

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

WAIT_TIMEOUT = 4
DEFAULT_LIMIT = 2000000000


@pytest.fixture(scope="module")
def cases():
    make = {"qwen": workloads.qwen3_8b, "gptoss": workloads.gpt_oss_20b}
    return {(n, s): Case(make[n](batch=1, seq_len=1024, calib_tokens=2048, lloyd_iters=4), key_scale=s)
            for n in make for s in (False, True)}


@pytest.mark.parametrize("n", [300, 4099])
@pytest.mark.parametrize("name,fmt", [("qwen", "plain"), ("gptoss", "plain"), ("qwen", "scaled"), ("qwen", "deployed"),
                                      ("gptoss", "deployed")])
def test_waits_that_give_up(cases, name, fmt, n):
    from paper_2608_04074_b200.runtime import PagedCache
    case = cases[name, fmt != "plain"]
    ctx = case.ctx
    cache = PagedCache(ctx, np.zeros(2, np.int32), capacity_tokens=np.array([n, 640], np.int32), seed=11,
                       key_scale=fmt == "scaled", int2_values=fmt == "deployed")
    pools = [x for x in (cache.k_pages, cache.v_pages, cache.k_scales, cache.v_meta) if x is not None]
    k, v, _ = case.draw(5000, n, 1)
    dev = lambda a, dtype=torch.int32: torch.from_numpy(np.ascontiguousarray(a)).to(dtype).cuda()
    args = (dev(k, torch.bfloat16), dev(v, torch.bfloat16), dev(np.zeros(n)), dev(np.arange(n)))
    own = torch.zeros(cache.n_pages, dtype=torch.bool, device="cuda")
    own[dev(cache.page_table_host[0][: (n + 63) // 64], torch.int64)] = True

    cache.append(0, *args)
    assert ctx.novakv_last_device_status() == 0
    expected = [x.clone() for x in pools]
    seen = 0
    try:
        for limit in (0, 1, 2, 3, 5, 8, 16, 32, 100, 500, 0):
            ctx.novakv_debug_set_wait_limit(limit)
            for p in pools:
                p[~own] = 0x5a if p.dtype == torch.uint8 else 3.0
            cache.append(0, *args)
            status = ctx.novakv_last_device_status()
            assert status in (0, WAIT_TIMEOUT)
            assert limit > 0 or status == WAIT_TIMEOUT
            seen += status != 0
            for p, e in zip(pools, expected):
                assert bool((p[~own] == (0x5a if p.dtype == torch.uint8 else 3.0)).all())
                if status == 0:
                    assert torch.equal(p[own], e[own])
            assert int(cache.seq_lens[1]) == 0
    finally:
        ctx.novakv_debug_set_wait_limit(DEFAULT_LIMIT)
    assert seen
    cache.append(0, *args)
    assert ctx.novakv_last_device_status() == 0
    for p, e in zip(pools, expected):
        assert torch.equal(p[own], e[own])
