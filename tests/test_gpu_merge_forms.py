"""The forms of the prepare and merge kernels on both sides of the batch sizes at which they change: one sequence per block (at
most as many pairs as SMs), one per block in half the registers (eight heads per KV head, beyond that), runs of sequences in
the merge kernel (up to four heads, beyond that) and in the prepare kernel (more pairs than two per SM) - with and without a
sink logit, with empty sequences first, last and inside a run.  Bound: 2e-3 of the largest output (check_output)."""
import numpy as np
import pytest

from gpu_common import Case, check_output
from paper_2608_04074_b200 import workloads

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def cases():
    return {"qwen": Case(workloads.qwen3_8b(batch=1, seq_len=1024, calib_tokens=2048, lloyd_iters=4)),
            "gptoss": Case(workloads.gpt_oss_20b(batch=1, seq_len=1024, calib_tokens=2048, lloyd_iters=4))}


@pytest.mark.parametrize("sink", [False, True])
@pytest.mark.parametrize("edge", ["one_per_sm", "more", "two_per_sm", "runs"])
@pytest.mark.parametrize("name", ["qwen", "gptoss"])
def test_batches_around_the_lines(cases, name, edge, sink):
    from paper_2608_04074_b200.runtime import PagedCache
    case = cases[name]
    hkv, n_sm = case.ctx.n_kv_heads, torch.cuda.get_device_properties(0).multi_processor_count
    batch = {"one_per_sm": n_sm // hkv, "more": n_sm // hkv + 1, "two_per_sm": 2 * n_sm // hkv, "runs": 2 * n_sm // hkv + 1}[edge]
    lens = (37 * np.arange(batch) % 200).astype(np.int32)              # the first is empty
    lens[batch // 2] = lens[-1] = 0
    lens[1] = 1500                                                     # one with many pieces
    cache = PagedCache(case.ctx, lens, seed=9)
    k, v, _ = case.draw(6000, 1500, 1)
    e = case.oracle.encode(k.astype(np.float64), v.astype(np.float64), with_gaps=False)
    first = [11 * b % 1300 if n <= 200 else 0 for b, n in enumerate(lens)]
    part = [(e["kidx"][f:f + n], e["vidx"][f:f + n]) for f, n in zip(first, lens)]
    cache.store_logical_batch([(b, 0, *p) for b, p in enumerate(part) if lens[b]])
    _, _, q = case.draw(6001, 1, batch)
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
