"""The measurement entry points of the C ABI (loopspec_time_kernel, loopspec_launches_per_step, loopspec_decode_paths):
they run, report what the header says, leave the context usable, and what they report matches what a decode step does."""
import numpy as np
import pytest

from tests import gpu_util as U
import workloads as W

pytestmark = pytest.mark.gpu


def test_decode_paths_follow_the_row_and_context_capacity():
    """Passes of up to 8 rows: mma.sync cluster kernels; 9 to 64 rows of a bf16 model: the tcgen05 kernel + epilogue;
    attention_path tells a long context capacity: beyond 2560 positions, 512 when the context holds several sequences;
    fp32 weights never leave the CUDA cores."""
    cases = [(dict(name="tiny_bf16", max_seqs=1, max_ctx=256), (0, 0)),
             (dict(name="tiny_bf16", max_seqs=4, max_ctx=256), (1, 0)),
             (dict(name="tiny_bf16", max_seqs=1, max_ctx=1001), (0, 0)),
             (dict(name="tiny_bf16", max_seqs=1, max_ctx=2560), (0, 0)),
             (dict(name="tiny_bf16", max_seqs=1, max_ctx=2561), (0, 1)),
             (dict(name="tiny_bf16", max_seqs=1, max_ctx=3000), (0, 1)),
             (dict(name="tiny_bf16", max_seqs=4, max_ctx=1024), (1, 1)),
             (dict(name="tiny_bf16", max_seqs=4, max_ctx=512), (1, 0)),
             (dict(name="tiny_raven", max_seqs=1, max_ctx=256), (1, 0)),
             (dict(name="tiny", max_seqs=4, max_ctx=256), (0, 0))]
    for kw, want in cases:
        shape = W.CONFIGS[kw["name"]]
        d1, d2 = (2, 8) if shape.R >= 16 else (1, 2)
        ctx = U.make_ctx(kw["name"], d1, d2, max_seqs=kw["max_seqs"], max_ctx=kw["max_ctx"])
        assert ctx.decode_paths() == want, (kw, ctx.decode_paths())
        ctx.close()


def test_launch_count_matches_the_kernels_of_a_pass():
    """1 preparation + 5 kernels per block + lm_head + selection + control + KV commit for passes of up to 8 rows;
    two launches per GEMM on the tcgen05 path."""
    shape = W.CONFIGS["tiny_bf16"]
    ctx = U.make_ctx("tiny_bf16", 1, 2, max_seqs=1, max_ctx=128)
    assert ctx.launches_per_step() == 1 + 5 * shape.n_recurrent + 4
    ctx.close()
    ctx = U.make_ctx("tiny_bf16", 1, 2, max_seqs=4, max_ctx=128)
    assert ctx.launches_per_step() == 1 + 9 * shape.n_recurrent + 4
    ctx.close()


@pytest.mark.parametrize("max_ctx", [512, 3000])
def test_kernels_can_be_timed_alone_and_the_context_stays_usable(max_ctx):
    """Every kernel of the pass through loopspec_time_kernel: sane times, the byte counts of the header's formulas, and
    a decode after a new prefill still matches the oracle."""
    name = "tiny_bf16"
    shape = W.CONFIGS[name]
    ref = U.oracle_run(name, 20, 12, 1, 2, T=1.0, seed=5)
    ctx = U.make_ctx(name, 1, 2, T=1.0, seed=5, max_seqs=2, max_ctx=max_ctx, max_prefill_rows=32)
    assert ctx.prefill(ref["prompt"]) == ref["first"]
    hq, hkv = shape.n_q_heads * shape.head_dim, shape.n_kv_heads * shape.head_dim
    wbytes = [(hq + 2 * hkv) * shape.hidden * 2, shape.hidden * hq * 2, 2 * shape.ffn * shape.hidden * 2, shape.hidden * shape.ffn * 2,
              shape.vocab * shape.hidden * 2]
    for which in range(5):
        ms, nbytes = ctx.time_kernel(which, 4, 5)
        assert 0 < ms < 5.0 and nbytes == wbytes[which]
    kv_ctx = 2 * hkv * (max_ctx - 64) * 2
    ms, nbytes = ctx.time_kernel(5, 6, 5)           # decode attention: every row a context of its own
    assert 0 < ms < 50.0 and nbytes == 6 * kv_ctx
    ms, nbytes = ctx.time_kernel(6, 32, 5)          # prefill attention: the rows share one context
    assert 0 < ms < 50.0 and nbytes == kv_ctx
    with pytest.raises(Exception):
        ctx.time_kernel(6, 33, 1)                   # more rows than a prefill pass carries
    with pytest.raises(Exception):
        ctx.decode(4)                               # the timed launches used the sequences' state: a prefill comes first
    assert ctx.prefill(ref["prompt"]) == ref["first"]
    ctx.decode(12)
    U.assert_same_run(ctx, ref, 12)
    ctx.close()


@pytest.mark.parametrize("which", [0, 2, 3])
def test_a_timed_wide_gemm_finishes_every_row_whatever_bounds_a_prefill_pass(which):
    """The timed launches run in the decode launch configuration: with prefill passes of at most 16 rows, 24 rows of a GEMM on the
    tcgen05 path write as much of the workspace as with passes of 64 (the two contexts are otherwise in the same state)."""
    import torch
    name, S = "tiny_bf16", 8
    refs = [U.oracle_run(name, 16, 12, 1, 2, seq=s) for s in range(S)]
    changed = []
    for rows_pf in (16, 64):
        ctx = U.make_ctx(name, 1, 2, max_seqs=S, max_ctx=64, max_prefill_rows=rows_pf)
        for s in range(S):
            assert ctx.prefill(refs[s]["prompt"], seq=s) == refs[s]["first"]
        ctx.decode(12)
        assert ctx.decode_paths()[0] == 1 and ctx.stats()["rows_max"] >= 24
        ctx.time_kernel(1, 24, 1)                       # the scratch table and states of the timed launches are in place
        torch.cuda.synchronize()
        before = ctx.workspace.clone()
        ctx.time_kernel(which, 24, 1)
        torch.cuda.synchronize()
        n = before.numel() // 4 * 4
        changed.append(int((before[:n].view(torch.int32) != ctx.workspace[:n].view(torch.int32)).sum()))
        ctx.close()
    assert changed[0] == changed[1], changed
