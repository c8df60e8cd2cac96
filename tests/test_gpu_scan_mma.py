"""Decode of the d = 64 shape with eight query heads per KV head (logits on tensor cores): ragged lengths around the
32-token tiles, the 64-token pages and the 16 warps' 512-token stride, and query magnitudes over the range in which the
binary16 halves of the scaled query must neither overflow nor vanish.

Bound: the weights are rounded to binary16 (2^-11 each, both in the sum and in the normaliser), the value grid has 7 bits
and the logits are good to 3e-7, so the outputs stay well within the 2e-3 of check_output."""
import numpy as np
import pytest

from gpu_common import Case, check_output
from paper_2608_04074_b200 import workloads

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def case():
    return Case(workloads.gpt_oss_20b(batch=2, seq_len=2048, calib_tokens=4096, lloyd_iters=6))


# The tensor-core kernel is taken from a capacity of 5 pages (of 64 tokens) per SM on; the calls below it take the score table.
# `wide`: the smallest page table that reaches the first, and the largest that stays with the second.
@pytest.mark.parametrize("wide", [True, False], ids=["products", "table"])
@pytest.mark.parametrize("factor", [1.0, 16.0, 1e-3, 1e-30])
@pytest.mark.parametrize("lens", [[1], [31, 32, 33, 0, 63, 64, 65], [511, 512, 513, 1025], [3000], list(range(1, 160, 4))],
                         ids=lambda x: f"{len(x)}x{max(x)}")
def test_logits_on_tensor_cores(case, lens, factor, wide):
    from paper_2608_04074_b200.runtime import PagedCache
    need, per_page = 5 * torch.cuda.get_device_properties(0).multi_processor_count, len(lens) * case.ctx.n_kv_heads
    pages = -(-need // per_page) - (0 if wide else 1)
    assert wide == (pages * per_page >= need)
    if 64 * pages < max(lens):
        pytest.skip("so many sequences of this length are past the line whatever the capacity")
    cap = np.array(lens, np.int32)
    cap[0] = 64 * pages                                       # (the table is as wide as its longest row)
    cache = PagedCache(case.ctx, np.array(lens, np.int32), capacity_tokens=cap, seed=5)
    assert cache.page_table.shape[1] == pages
    encs, items = [], []
    for b, n in enumerate(lens):
        k, v, _ = case.draw(700 + b, max(n, 1), 1)
        e = case.oracle.encode(k.astype(np.float64), v.astype(np.float64), with_gaps=False)
        encs.append(e)
        if n:
            items.append((b, 0, e["kidx"], e["vidx"]))
    cache.store_logical_batch(items)
    _, _, q = case.draw(701, 1, len(lens))
    q[:, 3] = 0.0                                             # one head without a direction: the mean of the values
    scale = factor / np.sqrt(case.ctx.head_dim)
    out = cache.decode(0, torch.from_numpy(q).to(torch.bfloat16).cuda(), sm_scale=scale).cpu().numpy()
    assert case.ctx.novakv_last_device_status() == 0
    for b, n in enumerate(lens):
        if n == 0:
            assert not out[b].any()
        else:
            check_output(out[b], case.oracle.decode(q[b].astype(np.float64), encs[b]["kidx"], encs[b]["vidx"], sm_scale=scale))


def test_no_further_from_binary64_than_the_table_kernel(case):
    """The halves of query and codewords and the tensor core's truncation must not cost what the binary32 score table had: the
    output error against binary64 stays within that of the table kernel (reached by the fused merge) on the same cache.  The
    weights are binary16 numbers in both, and round alike: the two errors are equal to a percent (1.03 with eight chained
    products per logit and the grid's centre removed afterwards)."""
    from paper_2608_04074_b200.runtime import PagedCache
    lens = np.full(24, 700, np.int32)
    cache = PagedCache(case.ctx, lens, seed=5)
    encs = [case.oracle.encode(*(x.astype(np.float64) for x in case.draw(900 + b, 700, 1)[:2]), with_gaps=False) for b in range(24)]
    cache.store_logical_batch([(b, 0, e["kidx"], e["vidx"]) for b, e in enumerate(encs)])
    _, _, q = case.draw(901, 1, 24)
    scale = case.ctx.head_dim ** -0.5
    refs = np.stack([case.oracle.decode(q[b].astype(np.float64), e["kidx"], e["vidx"], sm_scale=scale) for b, e in enumerate(encs)])
    err = {}
    try:
        for fused in (False, True):
            case.ctx.novakv_debug_set_fused_merge(fused)
            err[fused] = np.linalg.norm(cache.decode(0, torch.from_numpy(q).to(torch.bfloat16).cuda(), sm_scale=scale).cpu().numpy() - refs)
    finally:
        case.ctx.novakv_debug_set_fused_merge(False)
    assert err[False] <= 1.01 * err[True], err[False] / err[True]
