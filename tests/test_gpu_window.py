"""Sliding-window / short-capacity decode on the BF16 cache where one CTA has a sequence to itself and writes the output
(at most 16 pages), next to the first size that is split (17 pages): windows that start inside a group of 8 tokens, inside a
page and before the sequence.  Reference and bound: the parity suite's (textbook attention, 2e-3 of the largest output)."""
import numpy as np
import pytest

from gpu_common import Case, check_output
from oracle import novakv_oracle as O
from paper_2608_04074_b200 import synth, workloads

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def cases():
    return {"qwen": Case(workloads.qwen3_8b(batch=1, seq_len=1024, calib_tokens=2048, lloyd_iters=4)),
            "gptoss": Case(workloads.gpt_oss_20b(batch=1, seq_len=1024, calib_tokens=2048, lloyd_iters=4))}


@pytest.mark.parametrize("dtype", [torch.float32, torch.bfloat16])
@pytest.mark.parametrize("window,lens", [(1, [1, 64, 65]), (127, [5, 128, 191, 0, 700]), (130, [1023, 131]), (961, [1000, 1088]),
                                         (962, [1000, 1088]), (960, [1087, 1023]), (961, [1026, 1087]), (962, [1026, 1087]),
                                         (0x7fffffff, [1088, 7]), (0, [1024, 3, 0]), (0, [1025, 9]),
                                         (127, [5, 128, 191, 0, 700, *range(120, 140)])])     # more CTAs than SMs: four warps each
@pytest.mark.parametrize("name", ["qwen", "gptoss"])
def test_one_cta_per_sequence(cases, name, window, lens, dtype):
    case, lens = cases[name], np.array(lens, np.int32)
    ctx, dev = case.ctx, (lambda a: torch.from_numpy(np.ascontiguousarray(a)).cuda())
    table, n_pages = synth.shuffled_page_table(7, np.maximum(lens, 1), 64)
    kp = np.full((n_pages, ctx.n_kv_heads, 64, ctx.head_dim), np.nan, np.float32)      # bytes past a sequence are arbitrary
    vp = kp.copy()
    rows = []
    for b, n in enumerate(lens):
        k, v, _ = case.draw(1500 + b, max(int(n), 1), 1)
        rows.append((k[:n], v[:n]))
        pos = np.arange(n)
        kp[table[b][pos // 64], :, pos % 64, :] = k[:n]
        vp[table[b][pos // 64], :, pos % 64, :] = v[:n]
    _, _, q = case.draw(1550, 1, len(lens))
    ws = torch.empty(ctx.novakv_bf16_workspace_bytes(len(lens), table.shape[1]), dtype=torch.uint8, device="cuda")
    out = torch.full((len(lens), ctx.n_q_heads, ctx.head_dim), float("nan"), dtype=dtype, device="cuda")
    before = ctx.novakv_launch_count()
    ctx.novakv_bf16_decode_attention(dev(q).to(torch.bfloat16), dev(kp).to(torch.bfloat16), dev(vp).to(torch.bfloat16),
                                     dev(np.where(table < 0, 0, table).astype(np.int32)), dev(lens), out, ws, window=window)
    # one kernel while 16 pages hold the capacity, or the window wherever it ends; else a merge kernel follows
    assert ctx.novakv_launch_count() - before == (1 if table.shape[1] <= 16 or 0 < window <= 961 else 2)
    got = out.float().cpu().numpy()
    for b, n in enumerate(lens):
        if n == 0:
            assert not got[b].any()
            continue
        k, v = (x[max(0, int(n) - window) if window else 0:].astype(np.float64) for x in rows[b])
        ref = O.attention(q[b].astype(np.float64), k, v)
        if dtype == torch.bfloat16:                          # 2^-9 of each output (<= 1.96e-3 of the largest) on top
            assert np.abs(got[b] - ref).max() <= (2e-3 + 2.0 ** -9) * np.abs(ref).max()
        else:
            check_output(got[b], ref)
