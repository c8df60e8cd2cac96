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


@pytest.mark.parametrize("factor", [1.0, 16.0, 1e-3, 1e-30])
@pytest.mark.parametrize("lens", [[1], [31, 32, 33, 0, 63, 64, 65], [511, 512, 513, 1025], [3000], list(range(1, 160, 4))],
                         ids=lambda x: f"{len(x)}x{max(x)}")
def test_logits_on_tensor_cores(case, lens, factor):
    from paper_2608_04074_b200.runtime import PagedCache
    cache = PagedCache(case.ctx, np.array(lens, np.int32), seed=5)
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
